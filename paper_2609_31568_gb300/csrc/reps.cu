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
constexpr int kBand = 4096;       // cosines of a chunk that the clustering keeps in shared memory

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
    float* gram;
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
// a launch covers. IN: loads in flight of a thread.
template <int IN>
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
        for (; t + (IN - 1) * kFpWarps < t1; t += IN * kFpWarps) {
            uint4 x[IN];
#pragma unroll
            for (int u = 0; u < IN; ++u) x[u] = ld_stream(src + (t + u * kFpWarps) * D8);
#pragma unroll
            for (int u = 0; u < IN; ++u) add_bf16x8(acc, x[u]);
        }
        if (t < t1) {
            uint4 x[IN - 1];
#pragma unroll
            for (int u = 0; u < IN - 1; ++u)
                x[u] = t + u * kFpWarps < t1 ? ld_stream(src + (t + u * kFpWarps) * D8) : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int u = 0; u < IN - 1; ++u) add_bf16x8(acc, x[u]);
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

// Exclusive block scan of the threads' counts; returns this thread's exclusive
// prefix, *total receives the block total.
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

// Algorithm 1 in outer chunk c: the anchor a admits j while cos(v_a, v_j) >= theta
// and |C_a| < S_max. The walk is a chain of dependent cosines. By one thread, with
// `band` the chunk's cosines in shared memory: 30 cycles a link instead of 700.
__device__ void walk_band(const StepArgs& a, int c, const float* band)
{
    const int c0 = c * a.per_outer, c1 = min(a.M, c0 + a.per_outer);
    for (int an = c0; an < c1;) {
        a.flag[an] = 1;
        int j = an + 1;
        for (; j < c1 && j - an < a.S_max && band[(an - c0) * a.S_max + j - an] >= a.theta; ++j) a.flag[j] = 0;
        an = j;
    }
}

// By the CTA, with the cosines of as many sub-chunks at a time as shared memory
// holds: step (a) of 512K tokens of 4 heads on one, an outer chunk of 4,096
// sub-chunks and each a cluster, takes 552 us (a load per link: 1,543).
__device__ void walk_windows(const StepArgs& a, int c, float* band, int* next)
{
    const int c1 = min(a.M, (c + 1) * a.per_outer), S_max = a.S_max;
    for (int an = c * a.per_outer; an < c1;) {
        const int rows = min(c1 - an, kBand / S_max);
        const float* src = a.gram + static_cast<int64_t>(an) * S_max;
#pragma unroll 4
        for (int x = threadIdx.x; x < rows * S_max; x += blockDim.x) band[x] = __ldcg(src + x);
        __syncthreads();
        if (threadIdx.x == 0) {
            int at = an;
            while (at < an + rows) {
                a.flag[at] = 1;
                int j = at + 1;
                for (; j < c1 && j - at < S_max && band[(at - an) * S_max + j - at] >= a.theta; ++j) a.flag[j] = 0;
                at = j;
            }
            *next = at;
        }
        __syncthreads();
        an = *next;
        __syncthreads();
    }
}

// By one warp, a lane per candidate of the anchor, with the cosines in memory:
// clusters that may be longer than shared memory.
__device__ void walk_rows(const StepArgs& a, int c)
{
    const int lane = threadIdx.x & 31, c0 = c * a.per_outer, c1 = min(a.M, c0 + a.per_outer);
    for (int an = c0; an < c1;) {
        const int most = c1 - an < a.S_max ? c1 - an : a.S_max;
        int size = 1;
        for (int d0 = 1; d0 < most; d0 += 32) {
            const int d = d0 + lane;
            const float cs = d < most ? __ldcg(&a.gram[static_cast<int64_t>(an) * a.S_max + d]) : 0.f;
            const unsigned out = __ballot_sync(0xFFFFFFFFu, d >= most || !(cs >= a.theta));
            size = d0 + (out ? __ffs(out) - 1 : 32);
            if (out) break;
        }
        for (int i = lane; i < size; i += 32) a.flag[an + i] = i == 0;
        an += size;
    }
}

// The anchors of the outer chunks [c_begin, c_end) into unit_start, after the
// *n_units units of the chunks before c_begin, by one CTA: every thread a run of
// sub-chunks, counted, and after one scan written. `full`: every cluster takes
// S_max sub-chunks or what its outer chunk has left.
__device__ void compact(const StepArgs& a, bool full, int* sh)
{
    const int M = a.M, m_begin = a.c_begin * a.per_outer, m_end = min(M, a.c_end * a.per_outer);
    // read before the first barrier; thread 0 rewrites it after the last
    const int offset = a.c_begin == 0 ? 0 : *a.n_units;
    const int run = (m_end - m_begin + static_cast<int>(blockDim.x) - 1) / static_cast<int>(blockDim.x);
    const int r0 = m_begin + static_cast<int>(threadIdx.x) * run, r1 = min(m_end, r0 + run);
    auto is_anchor = [&](int i) { return full ? i % a.per_outer % a.S_max == 0 : __ldcg(&a.flag[i]) != 0; };
    int count = 0, total;
    uint32_t first = 0;  // the run's first 32 are read once
#pragma unroll 4
    for (int i = r0; i < r1; ++i) {
        const uint32_t f = is_anchor(i);
        count += f;
        if (i - r0 < 32) first |= f << (i - r0);
    }
    int at = offset + block_exclusive_scan(count, sh, &total);
    for (int i = r0; i < r1; ++i)
        if (i - r0 < 32 ? first >> (i - r0) & 1u : is_anchor(i)) a.unit_start[at++] = i;
    for (int i = offset + total + static_cast<int>(threadIdx.x); i <= M; i += blockDim.x) a.unit_start[i] = M;
    if (threadIdx.x == 0) *a.n_units = offset + total;
}

// Arrivals at the clusters of outer chunk c, counted in the unused cosine of its
// first sub-chunk with itself.
__device__ __forceinline__ int32_t* chunk_ticket(const StepArgs& a, float* gram, int c)
{
    return reinterpret_cast<int32_t*>(gram + static_cast<int64_t>(c) * a.per_outer * a.S_max);
}

// gram[i][d] = cos(v_i, v_{i+d}) = v~_i . v~_{i+d} for 1 <= d < S_max and i+d
// in the same outer chunk; 0 when either norm is 0. One warp per (i, d);
// `rows` neighbouring i of one outer chunk per CTA. Where the cosines of all
// chunks fit shared memory, the CTA that finishes last (a ticket that k_step_a
// cleared) walks and compacts the clusters of all of them; else the last one of
// every chunk walks the chunk and the last one of these compacts. Step (a) of 4K
// tokens of one head in 32 sub-chunks: 12.5 us (19 with a ticket per chunk); of 1M
// tokens in 8,192: 169 us (all chunks walked by the last CTA 608 us).
__global__ void __launch_bounds__(512) k_gram(const StepArgs args, float* __restrict__ gram, int rows)
{
    __shared__ int sh[40];
    __shared__ int last;
    __shared__ float band[kBand];
    scale_ptx::pdl_enter();
    const float* fp = args.fp;
    const float* ss_part = args.ss_part;
    const int groups = args.fp_groups, D = args.D8 * 8, M = args.M, S_max = args.S_max, per_outer = args.per_outer;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nw = blockDim.x >> 5;
    const int ctas = (per_outer + rows - 1) / rows;  // of a full chunk
    const int c = args.c_begin + static_cast<int>(blockIdx.x) / ctas;
    const int chunk = c * per_outer, chunk_end = min(M, chunk + per_outer);
    const int i0 = chunk + static_cast<int>(blockIdx.x) % ctas * rows, i1 = min(chunk_end, i0 + rows);
    for (int x = warp; x < (i1 - i0) * (S_max - 1); x += nw) {
        const int i = i0 + (rows == 1 ? 0 : x / (S_max - 1)), d = x - (i - i0) * (S_max - 1) + 1, j = i + d;
        if (j >= chunk_end) continue;
        const float4* a = reinterpret_cast<const float4*>(fp + static_cast<int64_t>(i) * D);
        const float4* b = reinterpret_cast<const float4*>(fp + static_cast<int64_t>(j) * D);
        // 16-byte loads, four independent FMA chains (D is a multiple of 128)
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
#pragma unroll 8
        for (int e = lane; e < D / 4; e += 32) {
            const float4 u = a[e], v = b[e];
            s0 = fmaf(u.x, v.x, s0);
            s1 = fmaf(u.y, v.y, s1);
            s2 = fmaf(u.z, v.z, s2);
            s3 = fmaf(u.w, v.w, s3);
        }
        float s = (s0 + s1) + (s2 + s3);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
        const float na = fp_norm(ss_part, groups, i), nb = fp_norm(ss_part, groups, j);  // whole warp
        if (lane == 0) gram[static_cast<int64_t>(i) * S_max + d] = (na > 0.f && nb > 0.f) ? s / (na * nb) : 0.f;
    }
    // whether this CTA is the last of `of` to get here
    auto arrive = [&](int32_t* ticket, int of) {
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(ticket, 1) == of - 1;
        __syncthreads();
        __threadfence();
        return last != 0;
    };
    const int chunks = args.c_end - args.c_begin;
    const int64_t per_chunk = static_cast<int64_t>(per_outer) * S_max;
    const int held = per_chunk * chunks <= kBand ? chunks : 1;  // chunks that a CTA walks
    if (held == chunks) {
        if (!arrive(args.ticket, static_cast<int>(gridDim.x))) return;
    } else if (!arrive(chunk_ticket(args, gram, c), ctas)) {
        return;
    }
    const int cw = held == chunks ? args.c_begin : c;
    if (per_chunk <= kBand) {
        const int row0 = cw * per_outer, n = (min(M, (cw + held) * per_outer) - row0) * S_max;
#pragma unroll 4
        for (int x = threadIdx.x; x < n; x += blockDim.x) band[x] = __ldcg(gram + static_cast<int64_t>(row0) * S_max + x);
        __syncthreads();
        for (int x = threadIdx.x; x < held; x += blockDim.x) walk_band(args, cw + x, band + x * per_chunk);
        __syncthreads();
    } else if (S_max <= kBand) {
        walk_windows(args, cw, band, &last);
    } else if (warp == 0) {
        walk_rows(args, cw);
    }
    if (held < chunks && !arrive(args.ticket, chunks)) return;
    __syncthreads();
    compact(args, false, sh);
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
        if (a.theta <= -1.0f || a.S_max == 1) {
            compact(a, true, sh);
        } else {
            if (threadIdx.x == 0) *a.ticket = 0;
            for (int c = a.c_begin + static_cast<int>(threadIdx.x); c < a.c_end; c += kStepThreads)
                *chunk_ticket(a, a.gram, c) = 0;
        }
        return;
    }
    --x;
    if (x < a.nm * a.fp_groups) fingerprint<CTAS == 1 ? 16 : 8>(a, x / a.fp_groups, x % a.fp_groups, part, wsum);
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
    // 95.6 us (two per SM 88.7); even at 512. Where a second CTA per SM has little to
    // do a CTA's own loads decide: 16 in flight instead of 8 (2,689 tokens of 16
    // heads on 8 in sub-chunks of 2,048: 8.6 us, with 8 loads 10.3).
    const int64_t fps = static_cast<int64_t>(a.nm) * a.fp_groups;
    auto kern = pg.page_table ? k_step_a<true, 2>
                : grid <= sms ? k_step_a<false, 1>
                : d.L <= 512 && d.B <= 512 && fps > 2ll * sms ? k_step_a<false, 3> : k_step_a<false, 2>;
    e = launch_after(st, dim3(static_cast<unsigned>(grid)), kStepThreads, 0, 1, kern, a);
    if (e == cudaSuccess && d.S_max > 1 && d.theta > -1.0f) {
        // Several sub-chunks per CTA where there are many more than SMs for them;
        // a warp per cosine, and enough threads to compact the anchors.
        const int many = a.nm / (2 * sms);
        const int rows = many < 1 ? 1 : many < d.per_outer ? many : d.per_outer;
        const int64_t ctas = static_cast<int64_t>(c_end - c_begin) * ((d.per_outer + rows - 1) / rows);
        const int warps = d.S_max - 1 < 8 ? 8 : d.S_max - 1 < 16 ? d.S_max - 1 : 16;
        e = launch_after(st, dim3(static_cast<unsigned>(ctas)), 32 * warps, 0, 1, k_gram, a, gram, rows);
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
