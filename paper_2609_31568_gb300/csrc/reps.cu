// reps.cu -- step (a) of the SCR prefill path: block representative keys,
// sub-chunk fingerprints (Eq. 6) with their norms (Sec. V-A1), and
// anchor-based clustering (Eq. 8, Algorithm 1) inside each outer chunk.
//
// Two launches: k_step_a computes representatives and fingerprints side by
// side (and the clusters, where the threshold admits every sub-chunk), k_gram
// the cosines and then the clusters where the threshold decides. Both stream
// their inputs once with 16-byte loads and reduce in a fixed order, so their
// results are bit-reproducible run to run, and work on a range of outer chunks
// with the same per-element arithmetic as over the whole sequence.
#include <cuda_bf16.h>

#include "launch.cuh"
#include "ptx_sm103.cuh"
#include "scale_internal.h"

namespace scale {
namespace {

__device__ __forceinline__ void add_bf16x8(float (&acc)[8], const uint4 x)
{
    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        acc[2 * i] += __uint_as_float(w[i] << 16);
        acc[2 * i + 1] += __uint_as_float(w[i] & 0xFFFF0000u);
    }
}

__device__ __forceinline__ uint4 ld_stream(const uint4* p)
{
    uint4 r;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
                 : "l"(p));
    return r;
}

constexpr int kFpWarps = 16;
constexpr int kFpGroupCols = 32;  // sixteen-byte columns of a fingerprint CTA
constexpr int kStepThreads = 32 * kFpWarps;
constexpr int kBand = 4096;       // cosines that the clustering keeps in shared memory
static_assert(kBand * sizeof(float) <= kStepThreads * 2 * sizeof(float4), "k_step_a's buffer");

struct StepArgs {
    const uint4* q;
    const uint4* k;
    KvPaging pg;
    int64_t N;
    // fingerprints of the sub-chunks [m0, m0 + nm)
    int D8, L, nm, fp_groups;
    int64_t m0;
    float* fp;
    float* ss_part;
    // representatives of the blocks [b_base, b_end): `per` blocks of `groups` row
    // groups per CTA, row_cols sixteen-byte columns of a key row, `splits` CTAs
    // per row
    int row_chunks, row_cols, groups, per, splits, B;
    int64_t nb, b_base, b_end;
    float* reps;
    // clusters
    int M, S_max, per_outer, c_begin, c_end;
    float theta;
    const float* gram;
    int32_t* flag;
    int32_t* unit_start;
    int32_t* n_units;
    int32_t* ticket;
};

// Representative keys of `per` neighbouring blocks for every KV head: the means
// of the blocks' keys. Thread c of row group g of a block owns elements
// [8c, 8c + 8) of the token rows g, g + groups, ... of the block (every row read
// as one coalesced span), with 8 loads in flight; the groups' sums are then
// added in group order, so the result is bit-reproducible. Few KV heads and
// small blocks leave a block little to read: with 8 rows a group and as many
// blocks as the CTA has threads for, step (a) over 160K tokens of one query and
// one KV head takes 13.2 us in blocks of 64 (a block per CTA, 32 groups: 28.2 us).
template <bool PAGED>
__device__ void block_reps(const StepArgs& a, int item, float4* part)
{
    const int c = threadIdx.x % a.row_cols;
    const int x = threadIdx.x / a.row_cols;
    const int groups = a.groups, slot = x / groups, g = x - slot * groups;
    const int64_t b = a.b_base + static_cast<int64_t>(item / a.splits) * a.per + slot;
    const int col = item % a.splits * a.row_cols + c;
    const int64_t t0 = b * a.B;
    const int64_t t1 = (t0 + a.B < a.N) ? t0 + a.B : a.N;
    const bool live = slot < a.per && b < a.b_end && col < a.row_chunks;
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (live) {
        const uint4* src = a.k + col;
        const uint4 zero = make_uint4(0, 0, 0, 0);
        auto row = [&](int64_t t) {  // -1: a page outside the pool reads as zeros
            const int64_t r = PAGED ? kv_row(a.pg, t) : t;
            return PAGED && r < 0 ? zero : ld_stream(src + r * a.row_chunks);
        };
        int64_t t = t0 + g;
        for (; t + 7 * groups < t1; t += 8 * groups) {
            uint4 v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = row(t + i * groups);
#pragma unroll
            for (int i = 0; i < 8; ++i) add_bf16x8(acc, v[i]);
        }
        if (t < t1) {
            uint4 v[7];
#pragma unroll
            for (int i = 0; i < 7; ++i) v[i] = t + i * groups < t1 ? row(t + i * groups) : zero;
#pragma unroll
            for (int i = 0; i < 7; ++i) add_bf16x8(acc, v[i]);
        }
        part[(x * a.row_cols + c) * 2] = make_float4(acc[0], acc[1], acc[2], acc[3]);
        part[(x * a.row_cols + c) * 2 + 1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    }
    __syncthreads();
    if (g != 0 || !live) return;
    for (int gg = 1; gg < groups; ++gg) {
        const int y = (x + gg) * a.row_cols + c;
        const float4 lo = part[y * 2], hi = part[y * 2 + 1];
        acc[0] += lo.x; acc[1] += lo.y; acc[2] += lo.z; acc[3] += lo.w;
        acc[4] += hi.x; acc[5] += hi.y; acc[6] += hi.z; acc[7] += hi.w;
    }
    // acc held group 0's sum; the groups are added in order for every element
    const float cnt = static_cast<float>(t1 - t0);
    const int j = col / (kHeadDim / 8);
    const int d0 = (col % (kHeadDim / 8)) * 8;
    float4* dst = reinterpret_cast<float4*>(a.reps + (static_cast<int64_t>(j) * a.nb + b) * kHeadDim + d0);
    dst[0] = make_float4(acc[0] / cnt, acc[1] / cnt, acc[2] / cnt, acc[3] / cnt);
    dst[1] = make_float4(acc[4] / cnt, acc[5] / cnt, acc[6] / cnt, acc[7] / cnt);
}

// Fingerprint v_i (Eq. 6) of sub-chunk m0 + im, dimensions of one column
// group (32 sixteen-byte columns, i.e. 256 of the H_q * 128): the mean of its
// multi-head queries. Warp w sums the tokens w, w + 16, w + 32, ... of the
// sub-chunk for its lane's column, so every token row is read as one 512-byte
// span per warp; the 16 warps' sums are then added in warp order, divided by
// |X_i| and written, together with the group's sum of squares (the norm of
// Sec. V-A1 adds those in group order). The order is fixed, so the result is
// bit-reproducible and the same for a sub-chunk whichever range of sub-chunks
// a launch covers.
__device__ void fingerprint(const StepArgs& a, int im, int cg, float4* red, float* wsum)
{
    const int64_t i = a.m0 + im;
    const int D8 = a.D8;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int c = cg * kFpGroupCols + lane;
    const int64_t t0 = i * a.L;
    const int64_t t1 = (t0 + a.L < a.N) ? t0 + a.L : a.N;
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (c < D8) {
        const uint4* src = a.q + c;
        int64_t t = t0 + w;
        for (; t + 7 * kFpWarps < t1; t += 8 * kFpWarps) {
            uint4 x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = ld_stream(src + (t + u * kFpWarps) * D8);
#pragma unroll
            for (int u = 0; u < 8; ++u) add_bf16x8(acc, x[u]);
        }
        if (t < t1) {
            uint4 x[7];
#pragma unroll
            for (int u = 0; u < 7; ++u)
                x[u] = t + u * kFpWarps < t1 ? ld_stream(src + (t + u * kFpWarps) * D8) : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int u = 0; u < 7; ++u) add_bf16x8(acc, x[u]);
        }
    }
    red[(w * kFpGroupCols + lane) * 2] = make_float4(acc[0], acc[1], acc[2], acc[3]);
    red[(w * kFpGroupCols + lane) * 2 + 1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    __syncthreads();
    if (threadIdx.x < kFpGroupCols * 8) {
        // thread e owns element e of the group: column e / 8, lane e % 8 of it
        const int e = threadIdx.x;
        const float* flat = reinterpret_cast<const float*>(red);
        float v = 0.f;
        for (int ww = 0; ww < kFpWarps; ++ww) v += flat[ww * kFpGroupCols * 8 + e];
        v = v / static_cast<float>(t1 - t0);
        const int col = cg * kFpGroupCols + e / 8;
        float sq = 0.f;
        if (col < D8) {
            a.fp[i * static_cast<int64_t>(D8) * 8 + static_cast<int64_t>(col) * 8 + (e & 7)] = v;
            sq = v * v;
        }
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xFFFFFFFFu, sq, o);
        if (lane == 0) wsum[w] = sq;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int ww = 0; ww < kFpGroupCols * 8 / 32; ++ww) t += wsum[ww];
        a.ss_part[i * a.fp_groups + cg] = t;
    }
}

// ||v_i||_2 from the column groups' sums of squares, added in a fixed order
// (lane-strided, then a butterfly that leaves the same value in every lane).
// Warp-collective.
__device__ __forceinline__ float fp_norm(const float* __restrict__ ss_part, int groups, int i)
{
    const int lane = threadIdx.x & 31;
    float s = 0.f;
    for (int g = lane; g < groups; g += 32) s += ss_part[static_cast<int64_t>(i) * groups + g];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    return sqrtf(s);
}

// Exclusive block scan of 0/1 flags; returns this thread's exclusive prefix,
// *total receives the block total.
__device__ int block_exclusive_scan(int f, int* sh, int* total)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    int x = f;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        int run = 0;
        for (int i = 0; i < nw; ++i) {
            const int t = sh[i];
            sh[i] = run;
            run += t;
        }
        sh[nw] = run;
    }
    __syncthreads();
    const int excl = sh[w] + x - f;
    *total = sh[nw];
    __syncthreads();
    return excl;
}

// Algorithm 1 in the outer chunks [c_begin, c_end), by one CTA (one thread per
// chunk walks its sub-chunks: the anchor a admits j while cos(v_a, v_j) >=
// theta and |C_a| < S_max), which then compacts the anchor flags of those chunks
// into unit_start, after the *n_units units of the chunks before c_begin.
__device__ void cluster(const StepArgs& a, int* sh, float* band)
{
    const int M = a.M, S_max = a.S_max, per_outer = a.per_outer, c_begin = a.c_begin, c_end = a.c_end;
    const float theta = a.theta;
    int32_t* flag = a.flag;
    int32_t* unit_start = a.unit_start;
    int32_t* n_units = a.n_units;
    const bool always = theta <= -1.0f;
    // read before the first barrier; thread 0 rewrites it after the last
    int offset = c_begin == 0 ? 0 : *n_units;
    const int m_begin = c_begin * per_outer;
    const int m_end = min(M, c_end * per_outer);
    // cosine of sub-chunk an with sub-chunk j: cs(an, j - an)
    auto walk = [&](int c, auto cs) {
        const int c1 = min(M, (c + 1) * per_outer);
        int an = c * per_outer;
        while (an < c1) {
            flag[an] = 1;
            int size = 1, j = an + 1;
            while (j < c1 && size < S_max) {
                const bool admit = always || cs(an, j - an) >= theta;
                if (!admit) break;
                flag[j] = 0;
                ++size;
                ++j;
            }
            an = j;
        }
    };
    // The walk is a chain of dependent cosines: their band is brought into shared
    // memory, as many chunks at a time as fit (16 chunks of 16 sub-chunks: 30
    // cycles a link instead of 700).
    const int64_t per_chunk = static_cast<int64_t>(per_outer) * S_max;
    if (!always && per_chunk <= kBand) {
        const int batch = min(static_cast<int>(kBand / per_chunk), static_cast<int>(blockDim.x));
        for (int cb = c_begin; cb < c_end; cb += batch) {
            const int row0 = cb * per_outer;
            const int rows = min(m_end, (cb + batch) * per_outer) - row0;
            for (int i = threadIdx.x; i < rows * S_max; i += blockDim.x)
                band[i] = __ldcg(&a.gram[static_cast<int64_t>(row0) * S_max + i]);
            __syncthreads();
            const int c = cb + static_cast<int>(threadIdx.x);
            if (static_cast<int>(threadIdx.x) < batch && c < c_end)
                walk(c, [&](int an, int d) { return band[(an - row0) * S_max + d]; });
            __syncthreads();
        }
    } else {
        for (int c = c_begin + static_cast<int>(threadIdx.x); c < c_end; c += blockDim.x)
            walk(c, [&](int an, int d) { return __ldcg(&a.gram[static_cast<int64_t>(an) * S_max + d]); });
    }
    __syncthreads();
    for (int base = m_begin; base < m_end; base += blockDim.x) {
        const int i = base + threadIdx.x;
        const int f = (i < m_end) ? flag[i] : 0;
        int total;
        const int excl = block_exclusive_scan(f, sh, &total);
        if (f) unit_start[offset + excl] = i;
        offset += total;
    }
    for (int i = offset + threadIdx.x; i <= M; i += blockDim.x) unit_start[i] = M;
    if (threadIdx.x == 0) *n_units = offset;
}

// gram[i][d] = cos(v_i, v_{i+d}) = v~_i . v~_{i+d} for 1 <= d < S_max and i+d
// in the same outer chunk; 0 when either norm is 0. One warp per (i, d);
// one CTA per i in [m0, m0 + gridDim.x). The CTA that finishes last (a ticket
// that k_step_a cleared) then forms the clusters of the range.
__global__ void __launch_bounds__(512) k_gram(const StepArgs args, float* __restrict__ gram)
{
    __shared__ int sh[40];
    __shared__ int last;
    __shared__ float band[kBand];
    scale_ptx::pdl_enter();
    const float* fp = args.fp;
    const float* ss_part = args.ss_part;
    const int groups = args.fp_groups, D = args.D8 * 8, M = args.M, S_max = args.S_max, per_outer = args.per_outer;
    const int i = static_cast<int>(args.m0) + static_cast<int>(blockIdx.x);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nw = blockDim.x >> 5;
    const int chunk_end = min(M, (i / per_outer + 1) * per_outer);
    for (int d = warp + 1; d < S_max; d += nw) {
        const int j = i + d;
        if (j >= chunk_end) continue;
        const float4* a = reinterpret_cast<const float4*>(fp + static_cast<int64_t>(i) * D);
        const float4* b = reinterpret_cast<const float4*>(fp + static_cast<int64_t>(j) * D);
        // 16-byte loads, four independent FMA chains (D is a multiple of 128)
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 8
        for (int c = lane; c < D / 4; c += 32) {
            const float4 x = a[c], y = b[c];
            s0 = fmaf(x.x, y.x, s0);
            s1 = fmaf(x.y, y.y, s1);
            s2 = fmaf(x.z, y.z, s2);
            s3 = fmaf(x.w, y.w, s3);
        }
        float s = (s0 + s1) + (s2 + s3);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
        const float na = fp_norm(ss_part, groups, i), nb = fp_norm(ss_part, groups, j);  // whole warp
        if (lane == 0) gram[static_cast<int64_t>(i) * S_max + d] = (na > 0.f && nb > 0.f) ? s / (na * nb) : 0.f;
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(args.ticket, 1) == static_cast<int>(gridDim.x) - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    cluster(args, sh, band);
}

// Roles by CTA: the clusters where they need no cosine (one CTA), then the
// fingerprints, then the representatives, whose CTAs fill the SMs that the
// fingerprints of a short range leave free. Bound by HBM: 128K tokens of 32
// query and 8 KV heads (1.35 GB) with a threshold take 199 us with k_gram,
// 6.8 TB/s (222 us as four kernels); chunk by chunk with theta = -1 the eight
// calls of that layer take 0.25 ms less, a 4K layer's one call 14 us less.
template <bool PAGED, int CTAS>
__global__ void __launch_bounds__(kStepThreads, CTAS) k_step_a(const StepArgs a)
{
    __shared__ float4 part[kStepThreads * 2];
    __shared__ float wsum[8];
    __shared__ int sh[40];
    scale_ptx::pdl_enter();
    int x = blockIdx.x;
    if (x == 0) {
        if (threadIdx.x == 0) *a.ticket = 0;
        if (a.theta <= -1.0f || a.S_max == 1) cluster(a, sh, reinterpret_cast<float*>(part));
        return;
    }
    --x;
    if (x < a.nm * a.fp_groups) fingerprint(a, x / a.fp_groups, x % a.fp_groups, part, wsum);
    else block_reps<PAGED>(a, x - a.nm * a.fp_groups, part);
}

}  // namespace

int outer_chunks(const Derived& d)
{
    return static_cast<int>((d.M + d.per_outer - 1) / d.per_outer);
}

cudaError_t launch_build_reps_range(const Derived& d, const void* q, const void* k, const KvPaging& pg,
                                    float* reps, float* fingerprints, int32_t* unit_start,
                                    int32_t* n_units, int c_begin, int c_end, uint8_t* ws,
                                    cudaStream_t st)
{
    if (c_begin < 0 || c_end > outer_chunks(d) || c_begin >= c_end) return cudaSuccess;
    const WsLayout lay = ws_layout(d);
    float* ss_part = reinterpret_cast<float*>(ws + lay.fp_ss);
    float* gram = reinterpret_cast<float*>(ws + lay.gram);
    int32_t* flag = reinterpret_cast<int32_t*>(ws + lay.anchor);

    // Tokens [t0, t1) and sub-chunks [m0, m1) of the chunks. A block belongs to
    // the range holding its last token, so every key it averages is present
    // once the chunks up to this range are.
    const int64_t L_outer = static_cast<int64_t>(d.per_outer) * d.L;
    const int64_t t0 = c_begin * L_outer;
    const int64_t t1 = c_end * L_outer < d.N ? c_end * L_outer : d.N;
    const int64_t m0 = static_cast<int64_t>(c_begin) * d.per_outer;
    const int64_t m1 = static_cast<int64_t>(c_end) * d.per_outer < d.M ? static_cast<int64_t>(c_end) * d.per_outer
                                                                         : d.M;
    const int64_t b0 = t0 / d.B;
    const int64_t b1 = t1 == d.N ? d.nb : t1 / d.B;

    StepArgs a{};
    a.q = static_cast<const uint4*>(q);
    a.k = static_cast<const uint4*>(k);
    a.pg = pg;
    a.N = d.N;
    a.D8 = d.D / 8;
    a.L = d.L;
    a.nm = static_cast<int>(m1 - m0);
    a.fp_groups = d.fp_groups;
    a.m0 = m0;
    a.fp = fingerprints;
    a.ss_part = ss_part;
    a.row_chunks = d.Hkv * (kHeadDim / 8);
    a.row_cols = a.row_chunks < kStepThreads ? a.row_chunks : kStepThreads;
    const int slots = kStepThreads / a.row_cols;  // row groups of a CTA, eight rows or more each
    a.groups = d.B / 8 < slots ? (d.B / 8 > 0 ? d.B / 8 : 1) : slots;
    a.per = slots / a.groups;
    a.splits = (a.row_chunks + a.row_cols - 1) / a.row_cols;
    a.B = d.B;
    a.nb = d.nb;
    a.b_base = b0;
    a.b_end = b1;
    a.reps = reps;
    a.M = static_cast<int>(d.M);
    a.S_max = d.S_max;
    a.per_outer = d.per_outer;
    a.c_begin = c_begin;
    a.c_end = c_end;
    a.theta = d.theta;
    a.gram = gram;
    a.flag = flag;
    a.unit_start = unit_start;
    a.n_units = n_units;
    a.ticket = reinterpret_cast<int32_t*>(ws + kTicketOffset);

    // block size 1 may skip the representatives: token-level selection reads K itself
    const int64_t rep_ctas = reps && b1 > b0 ? (b1 - b0 + a.per - 1) / a.per * a.splits : 0;
    const int64_t grid = 1 + static_cast<int64_t>(a.nm) * a.fp_groups + rep_ctas;
    if (grid > 0x7FFFFFFFll) return cudaErrorInvalidConfiguration;
    int sms = 0;
    cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    // Three CTAs per SM keep HBM busy while short sub-chunks are summed up, with 40
    // registers instead of 64 for the loads in flight. 160K tokens of 28 heads on 4
    // in sub-chunks of 128: 196 us (two per SM 228); of 2,048, 60K tokens of 32 on 8:
    // 95.6 us (two per SM 88.7); even at 512.
    const bool dense = d.L <= 512 && static_cast<int64_t>(a.nm) * a.fp_groups > 2ll * sms;
    auto kern = pg.page_table ? k_step_a<true, 2> : dense ? k_step_a<false, 3> : k_step_a<false, 2>;
    e = launch_after(st, dim3(static_cast<unsigned>(grid)), kStepThreads, 0, 1, kern, a);
    if (e == cudaSuccess && d.S_max > 1 && d.theta > -1.0f) {
        // a warp per cosine, and enough threads to compact the anchors
        const int warps = d.S_max - 1 < 8 ? 8 : d.S_max - 1 < 16 ? d.S_max - 1 : 16;
        e = launch_after(st, dim3(static_cast<unsigned>(a.nm)), 32 * warps, 0, 1, k_gram, a, gram);
    }
    return e;
}

cudaError_t launch_build_reps(const Derived& d, const void* q, const void* k, const KvPaging& pg,
                              float* reps, float* fingerprints, int32_t* unit_start, int32_t* n_units,
                              uint8_t* ws, cudaStream_t st)
{
    return launch_build_reps_range(d, q, k, pg, reps, fingerprints, unit_start, n_units, 0,
                                   outer_chunks(d), ws, st);
}

}  // namespace scale
