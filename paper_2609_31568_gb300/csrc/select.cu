// select.cu -- steps (b) and (c) of the SCR prefill path: cluster-level
// retrieval with head soft-voting (Eq. 9, Sec. V-A3 "Selection function
// instantiation") over block representative keys, then a deterministic top-k.
//
//   k_logits  z[u][h][b] = sigma * v_a(u)^(h) . r_b^(h/g)   (tcgen05 MMA per KV head:
//             128 blocks x 64 (unit, head) rows; both fp32 operands split
//             into three bf16 parts, six part products accumulated in fp32)
//   k_stats   per (u, h): max_b z and 1 / sum_b exp(z - max) over the candidates
//   k_vote    score[u][b] = sum_h exp(z[u][h][b] - max) / sum   (heads in order)
//   k_topk    a radix select of the k-th largest key and an index-ordered
//             compaction (up to 4096 candidates in shared memory; in the
//             token-level selection with more than 64K candidates, the
//             multi-CTA form below): output ascending, ties to the lower b.
// Sequences of little selection work run in one kernel instead, k_select_few.
//
// Candidates of unit u are the blocks with a token in [n_sink, W_u),
// W_u = max(0, s_u - n_local): the contiguous range [b_lo, b_hi(u)).
#include <cuda_bf16.h>

#include <cmath>

#include "launch.cuh"
#include "ptx_sm103.cuh"
#include "scale_internal.h"

namespace scale {
namespace {

// exp(x) of x <= 0 for the factors that merge partial sums, within about an
// ulp where expf here is an approximation of two: x = n ln 2 + y, the Taylor
// series of e^y for |y| <= ln 2 / 2 (its next term is below 2^-27), times 2^n.
// With expf the scores were 3 % further from 64 bits than sums over one
// maximum (relative error 9.16e-8 against 8.90e-8 at 128K tokens; now 8.84e-8).
__device__ __forceinline__ float exp_factor(float x)
{
    if (!(x > -87.0f)) return x != x ? x : 0.f;
    const float n = rintf(x * 1.44269504f);
    const float y = fmaf(n, 1.90465432e-9f, fmaf(n, -0.693147182f, x));  // ln 2 in two parts
    float p = 1.0f / 5040.0f;
    p = fmaf(p, y, 1.0f / 720.0f);
    p = fmaf(p, y, 1.0f / 120.0f);
    p = fmaf(p, y, 1.0f / 24.0f);
    p = fmaf(p, y, 1.0f / 6.0f);
    p = fmaf(p, y, 0.5f);
    p = fmaf(p, y, 1.0f);
    p = fmaf(p, y, 1.0f);
    return p * __int_as_float((static_cast<int>(n) + 127) << 23);
}

struct SelArgs {
    Units ut;
    int sc_begin, sc_end;  // sub-chunk range of units to process
    int Hq, g;
    int64_t nb;
    int B, k, n_sink, n_local;
    float sigma;
    int scored;           // scores are asked for: also of units that take every candidate
    int32_t* status;      // device status word (bounded waits of k_logits)
    uint64_t timeout_ns;
};

__device__ __forceinline__ void cand_range(const SelArgs& a, int64_t s, int64_t* lo, int64_t* hi)
{
    const int64_t W = s - a.n_local > 0 ? s - a.n_local : 0;
    *lo = a.n_sink / a.B;                 // first block with (b+1)B > n_sink
    // one past the last block with bB < W (both below 2^31: a 32-bit division)
    *hi = (static_cast<uint32_t>(W) + static_cast<uint32_t>(a.B) - 1u) / static_cast<uint32_t>(a.B);
    if (*hi > a.nb) *hi = a.nb;
    if (*hi < *lo) *hi = *lo;
}

// Tensor-core logits. A CTA owns 128 blocks of one KV head j and walks a
// segment of the call's unit tiles (64 (unit, query head of j) rows: row
// ul * g + hl is head j g + hl of unit ul of the tile, the anchor's fingerprint
// slice). The representatives are the MMA's rows (TMEM lanes), so a warp stores
// 32 consecutive blocks of a logit row at a time; they are staged once per CTA,
// the fingerprint rows once per tile into one of two buffers. Both are fp32;
// every value x is split into three bf16 parts x1 + x2 + x3 = x exactly (x1 =
// bf16(x), x2 = bf16(x - x1), x3 = x - x1 - x2), written by the threads straight
// into the 128-byte-swizzled K-major layout of the MMA. The six part products
// a_i b_j with i + j <= 4 are exact in fp32 and are accumulated in fp32 in TMEM;
// the three dropped ones are below 2^-24 of |a| |b|. Only candidate blocks of
// each row's unit are written. Warp 0 lane 0 issues the MMAs (two accumulators
// of 64 columns), warps 1-8 store, warps 9-16 load and split the next tile: the
// three overlap, and what bounds the kernel is the staging of a tile. 256
// units x 4,096 blocks x 32 heads: 63 us (one CTA per tile, staging both
// operands each time and nothing overlapped: 185 us).
constexpr int kLtStageThreads = 256;
constexpr int kLtStoreThreads = 256;
constexpr int kLtThreads = 32 + kLtStoreThreads + kLtStageThreads;
constexpr int kLtRows = 64;                        // (unit, head) rows of a tile
constexpr int kLtWarpRows = 32;                    // of which a storing warp takes half
constexpr int kLtSeg = 8;                          // most tiles of a CTA
constexpr uint32_t kLtBPart = 128 * 128 * 2;       // one bf16 part of the representatives
constexpr uint32_t kLtAPart = kLtRows * 128 * 2;   // one bf16 part of a tile's rows
constexpr uint32_t kLtSmem = 3 * kLtBPart + 2 * 3 * kLtAPart + 1024;
static_assert(kLtSmem + kLtSeg * kLtRows * 8 + 1024 <= 227 * 1024, "logits shared memory");

// Two fp32 values as three packed bf16 pairs, x1 + x2 + x3 = x for each.
__device__ __forceinline__ void split_pair(float x, float y, uint32_t (&p)[3])
{
    p[0] = scale_ptx::pack_bf16x2(x, y);
    x -= __uint_as_float(p[0] << 16);
    y -= __uint_as_float(p[0] & 0xFFFF0000u);
    p[1] = scale_ptx::pack_bf16x2(x, y);
    p[2] = scale_ptx::pack_bf16x2(x - __uint_as_float(p[1] << 16), y - __uint_as_float(p[1] & 0xFFFF0000u));
}

// Four consecutive fp32 values of row r, columns [c, c + 4), into the three
// bf16 parts at `base` (part s at base + s * PART, of two 64-column halves): 8
// bytes per part, at the 128-byte-swizzled K-major position of (r, c).
template <uint32_t PART>
__device__ __forceinline__ void put_split4(uint8_t* base, int r, int c, float4 v)
{
    uint32_t lo[3], hi[3];
    split_pair(v.x, v.y, lo);
    split_pair(v.z, v.w, hi);
    const int hf = c >> 6, cc = c & 63;  // half, column in the half
    const uint32_t off = hf * (PART / 2) + (r >> 3) * 1024 + (r & 7) * 128 + ((((cc >> 3) ^ (r & 7))) << 4) +
                         (cc & 7) * 2;
#pragma unroll
    for (int s = 0; s < 3; ++s) *reinterpret_cast<uint2*>(base + s * PART + off) = make_uint2(lo[s], hi[s]);
}

struct LtBars {
    uint64_t a_full[2], a_empty[2];
    uint64_t d_full[2], d_empty[2];
    uint64_t drain;
};

__device__ __forceinline__ void lt_fail(volatile int* abort_flag, int32_t* status)
{
    *abort_flag = 1;
    record_status(status, SCALE_ERR_TIMEOUT);
}

__global__ void __launch_bounds__(kLtThreads, 1) k_logits(SelArgs a, int seg, const float* __restrict__ fp,
                                                          const float* __restrict__ reps,
                                                          float* __restrict__ logits)
{
    using namespace scale_ptx;
    extern __shared__ uint8_t smem_raw[];
    __shared__ LtBars bars;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    __shared__ int s_hi[kLtSeg * kLtRows], s_anchor[kLtSeg * kLtRows];  // of the segment's units
    pdl_enter();
    const int U = kLtRows / a.g;  // units per tile
    const int u_end = unit_lower_bound(a.ut, a.sc_end);
    const int u0 = unit_lower_bound(a.ut, a.sc_begin) + static_cast<int>(blockIdx.x) * seg * U;
    if (u0 >= u_end) return;
    const int n_u = (u_end - u0 < seg * U) ? u_end - u0 : seg * U;
    const int j = blockIdx.z;
    const int64_t b0 = static_cast<int64_t>(blockIdx.y) * 128;
    const int D = a.Hq * kHeadDim;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // The candidates [lo, hi(u)) of the units grow with u: the tiles before the
    // first unit with a candidate in [b0, b0 + 128) have nothing to do here.
    int64_t s, e, lo, hi;
    int anc;
    unit_range(a.ut, u0 + n_u - 1, &anc, &s, &e);
    cand_range(a, s, &lo, &hi);
    if (hi <= b0 || lo >= b0 + 128 || lo >= hi || (!a.scored && hi - lo <= a.k)) return;
    for (int i = tid; i < n_u; i += kLtThreads) {
        unit_range(a.ut, u0 + i, &anc, &s, &e);
        cand_range(a, s, &lo, &hi);
        s_hi[i] = static_cast<int>(hi);
        s_anchor[i] = anc;
    }
    __syncthreads();
    int first = 0;  // first unit with a candidate here (the last one has)
    for (int last = n_u - 1; first < last;) {
        const int mid = (first + last) >> 1;
        if (s_hi[mid] <= b0) first = mid + 1;
        else last = mid;
    }
    const int i0 = first / U, n_it = (n_u + U - 1) / U - i0;

    uint8_t* smem = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
    uint8_t* bbuf = smem;                 // representatives, three parts
    uint8_t* abuf = smem + 3 * kLtBPart;  // two buffers of three parts
    // the staging warps' rows of tile i; those of the first tile are on their way
    // while the representatives are staged
    constexpr int kPer = kLtRows * 32 / kLtStageThreads;
    const int t = tid - (kLtThreads - kLtStageThreads);
    float4 v[kPer];
    auto load_tile = [&](int tile) {
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int x = t + i * kLtStageThreads, r = x >> 5, c = (x & 31) * 4;
            const int ul = r / a.g, u = tile * U + ul;
            v[i] = ul < U && u < n_u
                       ? __ldg(reinterpret_cast<const float4*>(fp + static_cast<int64_t>(s_anchor[u]) * D +
                                                               (j * a.g + r - ul * a.g) * kHeadDim + c))
                       : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    if (t >= 0) load_tile(i0);
    // a warp reads one 512-byte row; eight rows per thread in flight
    for (int x0 = tid; x0 < 128 * 32; x0 += 8 * kLtThreads) {
        float4 vb[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int x = x0 + i * kLtThreads, r = x >> 5, c = (x & 31) * 4;
            vb[i] = x < 128 * 32 && b0 + r < a.nb
                        ? __ldg(reinterpret_cast<const float4*>(reps + (j * a.nb + b0 + r) * kHeadDim + c))
                        : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int x = x0 + i * kLtThreads;
            if (x < 128 * 32) put_split4<kLtBPart>(bbuf, x >> 5, (x & 31) * 4, vb[i]);
        }
    }
    fence_proxy_async_smem();
    if (tid == 0) {
        abort_flag = 0;
        for (int i = 0; i < 2; ++i) {
            mbar_init(&bars.a_full[i], kLtStageThreads);
            mbar_init(&bars.a_empty[i], 1);
            mbar_init(&bars.d_full[i], 1);
            mbar_init(&bars.d_empty[i], kLtStoreThreads);
        }
        mbar_init(&bars.drain, 1);
        fence_barrier_init();
    }
    if (warp == 0) {
        tmem_alloc(&tmem_slot, 128);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;
    if (warp == 0) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16_f32(128, kLtRows, 0);
            const uint64_t bd = sdesc_sw128(smem_addr(bbuf), 16, 1024);
            const uint64_t ad0 = sdesc_sw128(smem_addr(abuf), 16, 1024);
            // (A part, B part): the products a_i b_j with i + j <= 4 (parts from 1)
            constexpr int kPa[6] = {0, 0, 1, 0, 1, 2};
            constexpr int kPb[6] = {0, 1, 0, 2, 1, 0};
            bool ok = true;
            for (int it = 0; it < n_it; ++it) {
                const int st = it & 1;
                if (!mbar_wait_bounded(&bars.a_full[st], (it >> 1) & 1, a.timeout_ns, &abort_flag)) { ok = false; break; }
                if (it >= 2 && !mbar_wait_bounded(&bars.d_empty[st], ((it >> 1) - 1) & 1, a.timeout_ns, &abort_flag)) { ok = false; break; }
                tc_fence_after();
                const uint64_t ad = ad0 + st * (3 * kLtAPart >> 4);
#pragma unroll
                for (int i = 0; i < 6; ++i)
                    mma_ss_k128_ab<kLtBPart / 2, kLtAPart / 2>(tmem + st * kLtRows, bd + kPb[i] * (kLtBPart >> 4),
                                                               ad + kPa[i] * (kLtAPart >> 4), idesc, i > 0 ? 1u : 0u);
                mma_commit(&bars.d_full[st]);
                mma_commit(&bars.a_empty[st]);
            }
            if (!ok) {
                lt_fail(&abort_flag, a.status);
                mma_commit(&bars.drain);
                mbar_wait_bounded(&bars.drain, 0, a.timeout_ns, nullptr);
            }
        }
    } else if (warp <= kLtStoreThreads / 32) {
        // ------------------------------------------------------------ stores
        const int q = warp & 3;  // TMEM lane quarter this warp may access
        const int r0 = warp > 4 ? kLtWarpRows : 0;  // its rows of the tile
        const uint32_t lane_base = tmem + (static_cast<uint32_t>(q * 32) << 16) + r0;
        const int64_t b = b0 + q * 32 + lane;  // this thread's block
        const bool in = b >= a.n_sink / a.B;
        const int ul0 = r0 / a.g, left0 = a.g - (r0 - ul0 * a.g);
        for (int it = 0; it < n_it; ++it) {
            const int st = it & 1;
            if (!__all_sync(0xFFFFFFFFu, mbar_wait_bounded(&bars.d_full[st], (it >> 1) & 1, a.timeout_ns, &abort_flag))) {
                if (lane == 0) lt_fail(&abort_flag, a.status);
                break;
            }
            tc_fence_after();
            uint32_t z[kLtWarpRows];
            tmem_ld32(lane_base + st * kLtRows, z);
            tmem_ld_wait();
            tc_fence_before();
            mbar_arrive(&bars.d_empty[st]);
            int ul = (i0 + it) * U + ul0, left = left0;
            float* dst = logits + (static_cast<int64_t>(u0 + ul) * a.Hq + j * a.g + a.g - left) * a.nb + b;
            bool live = in && ul < n_u && ul < (i0 + it + 1) * U && b < s_hi[ul];
#pragma unroll
            for (int c = 0; c < kLtWarpRows; ++c) {
                if (live) *dst = a.sigma * __uint_as_float(z[c]);
                dst += a.nb;
                if (--left == 0) {  // the next unit's heads
                    left = a.g;
                    ++ul;
                    dst += static_cast<int64_t>(a.Hq - a.g) * a.nb;
                    live = in && ul < n_u && ul < (i0 + it + 1) * U && b < s_hi[ul];
                }
            }
        }
    } else {
        // ------------------------------------------------------------ staging
        for (int it = 0; it < n_it; ++it) {
            const int st = it & 1;
            if (it >= 2 && !mbar_wait_bounded(&bars.a_empty[st], ((it >> 1) - 1) & 1, a.timeout_ns, &abort_flag)) {
                lt_fail(&abort_flag, a.status);
                break;
            }
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                const int x = t + i * kLtStageThreads;
                put_split4<kLtAPart>(abuf + st * 3 * kLtAPart, x >> 5, (x & 31) * 4, v[i]);
            }
            fence_proxy_async_smem();
            mbar_arrive(&bars.a_full[st]);
            if (it + 1 < n_it) load_tile(i0 + it + 1);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, 128);
    }
}

// One warp per (unit, head): row max and 1 / sum of exp(z - max) over the candidates.
__global__ void __launch_bounds__(256) k_stats(SelArgs a, const float* __restrict__ logits,
                                               float* __restrict__ stats)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int u_first = unit_lower_bound(a.ut, a.sc_begin);
    const int u_end = unit_lower_bound(a.ut, a.sc_end);
    const int64_t uh = static_cast<int64_t>(blockIdx.x) * 8 + warp;
    const int u = u_first + static_cast<int>(uh / a.Hq);
    const int h = static_cast<int>(uh % a.Hq);
    if (u >= u_end) return;
    int anc;
    int64_t s, e, lo, hi;
    unit_range(a.ut, u, &anc, &s, &e);
    cand_range(a, s, &lo, &hi);
    if (lo >= hi) return;
    const float* z = logits + (static_cast<int64_t>(u) * a.Hq + h) * a.nb;
    // Eight loads in flight per lane; each lane still combines its values in
    // index order, so the result does not depend on the batching.
    constexpr int kIn = 8;
    float m = -INFINITY;
    for (int64_t b0 = lo + lane; b0 < hi; b0 += 32 * kIn) {
        float x[kIn];
#pragma unroll
        for (int i = 0; i < kIn; ++i) x[i] = b0 + 32 * i < hi ? z[b0 + 32 * i] : -INFINITY;
#pragma unroll
        for (int i = 0; i < kIn; ++i) m = fmaxf(m, x[i]);
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
    float sum = 0.f;
    for (int64_t b0 = lo + lane; b0 < hi; b0 += 32 * kIn) {
        float x[kIn];
#pragma unroll
        for (int i = 0; i < kIn; ++i) x[i] = b0 + 32 * i < hi ? z[b0 + 32 * i] : 0.f;
#pragma unroll
        for (int i = 0; i < kIn; ++i)
            if (b0 + 32 * i < hi) sum += expf(x[i] - m);
    }
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
    if (lane == 0) {
        stats[(static_cast<int64_t>(u) * a.Hq + h) * 2] = m;
        stats[(static_cast<int64_t>(u) * a.Hq + h) * 2 + 1] = 1.0f / sum;
    }
}

// score[u][b] = sum over heads (in order) of exp(z - max) / sum; NaN off the candidates.
__global__ void __launch_bounds__(256) k_vote(SelArgs a, const float* __restrict__ logits,
                                              const float* __restrict__ stats,
                                              float* __restrict__ scores)
{
    const int u_first = unit_lower_bound(a.ut, a.sc_begin);
    const int u_end = unit_lower_bound(a.ut, a.sc_end);
    const int u = u_first + blockIdx.y;
    if (u >= u_end) return;
    const int64_t b = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (b >= a.nb) return;
    int anc;
    int64_t s, e, lo, hi;
    unit_range(a.ut, u, &anc, &s, &e);
    cand_range(a, s, &lo, &hi);
    float score = __int_as_float(0x7FC00000);
    if (b >= lo && b < hi) {
        score = 0.f;
        const float* zb = logits + static_cast<int64_t>(u) * a.Hq * a.nb + b;
        const float* sb = stats + static_cast<int64_t>(u) * a.Hq * 2;
        // Eight heads' loads in flight at a time, added in head order.
        constexpr int kIn = 8;
        for (int h0 = 0; h0 < a.Hq; h0 += kIn) {
            float z[kIn], mx[kIn], inv[kIn];
#pragma unroll
            for (int i = 0; i < kIn; ++i) {
                const int h = h0 + i < a.Hq ? h0 + i : a.Hq - 1;
                z[i] = zb[static_cast<int64_t>(h) * a.nb];
                mx[i] = sb[2 * h];
                inv[i] = sb[2 * h + 1];
            }
#pragma unroll
            for (int i = 0; i < kIn; ++i)
                if (h0 + i < a.Hq) score += expf(z[i] - mx[i]) * inv[i];
        }
    }
    scores[static_cast<int64_t>(u) * a.nb + b] = score;
}

// Order-preserving map of a float onto uint32 (larger float -> larger key).
__device__ __forceinline__ uint32_t float_key(float f)
{
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

constexpr int kTopkThreads = 1024;
constexpr int kSortMax = 4096;     // candidates up to which k_topk and k_select_fused keep the keys in shared memory

constexpr int kRadixBins = 2048;   // digits of 11, 11 and 10 bits
constexpr int kTopkPad = 128;
constexpr int kTopkCount = 256;    // keys up to which topk_emit counts instead

// Shared memory of topk_emit.
struct TopkShared {
    int hist[kRadixBins];
    int scan[32], gt[32], eq[32];
    int digit, need;
};

// The k picks among n > k > 0 keys in shared memory (candidate i is block
// lo + i), written to out in ascending order: a radix select of the k-th
// largest key T (three passes over the keys, each a histogram and one block
// scan of its bins), then the keys above T and the first ones equal to it, in
// index order (every warp owns a run of keys: counts, one scan, ballots).
// About 3 us for 1024 keys (the 55 exchange steps of a bitonic sort of 64-bit
// keys took 8). `keys` is 16-byte aligned, with room for kTopkPad more. Called
// by all THREADS threads of the CTA.
template <int THREADS>
__device__ void topk_emit(uint32_t* keys, int n, int64_t lo, int k, int32_t* out, TopkShared& sh)
{
    constexpr int kWarps = THREADS / 32;
    constexpr int kPer = kRadixBins / THREADS;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (n <= kTopkCount) {
        // Few keys: `per` threads per key count the keys ahead of it (larger, or
        // equal with a lower index); fewer than k make it a pick. The work grows
        // with n^2: against the three passes it saves 1.2 us per call at 250 keys,
        // 2 us at 60, and nothing at 500.
        int per = THREADS / kTopkCount;
        while (per < 32 && 2 * per * n <= THREADS) per *= 2;
        const int n_pad = (n + 4 * per - 1) / (4 * per) * (4 * per);
        if (tid < n_pad - n) keys[n + tid] = 0u;  // ahead of no key
        __syncthreads();
        const int i = tid / per, part = tid % per;
        const uint32_t mine = i < n ? keys[i] : 0u;
        int above = 0, level = 0;
#pragma unroll 4
        for (int x = 4 * part; x < n_pad; x += 4 * per) {
            const uint4 v = *reinterpret_cast<const uint4*>(keys + x);
            above += (v.x > mine) + (v.y > mine) + (v.z > mine) + (v.w > mine);
            level += (v.x >= mine) + (v.y >= mine) + (v.z >= mine) + (v.w >= mine);
        }
        for (int o = per / 2; o > 0; o >>= 1) {
            above += __shfl_xor_sync(0xFFFFFFFFu, above, o);
            level += __shfl_xor_sync(0xFFFFFFFFu, level, o);
        }
        if (__any_sync(0xFFFFFFFFu, i < n && level > above + 1)) {  // ties: the lower index first
            int ties = 0;
            for (int x = part; x < i && x < n; x += per) ties += keys[x] == mine;
            for (int o = per / 2; o > 0; o >>= 1) ties += __shfl_xor_sync(0xFFFFFFFFu, ties, o);
            above += ties;
        }
        const bool pick = i < n && above < k && part == 0;
        const unsigned b = __ballot_sync(0xFFFFFFFFu, pick);
        if (lane == 0) sh.scan[warp] = __popc(b);
        __syncthreads();
        int before = lane < warp ? sh.scan[lane] : 0;
        for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xFFFFFFFFu, before, o);
        if (pick) out[before + __popc(b & ((1u << lane) - 1u))] = static_cast<int32_t>(lo + i);
        return;
    }
    uint32_t prefix = 0;
    int need = k;
    for (int p = 0; p < 3; ++p) {
        const int shift = p == 0 ? 21 : p == 1 ? 10 : 0;
        const uint32_t mask = p == 2 ? 1023u : 2047u;
        for (int i = tid; i < kRadixBins; i += THREADS) sh.hist[i] = 0;
        __syncthreads();
        for (int i = tid; i < n; i += THREADS) {
            const uint32_t key = keys[i];
            // the digits above this one match (p == 0: all)
            if (p == 0 || (key >> (p == 1 ? 21 : 10)) == (prefix >> (p == 1 ? 21 : 10)))
                atomicAdd(&sh.hist[(key >> shift) & mask], 1);
        }
        __syncthreads();
        // the largest digit whose keys, with those above it, reach `need`:
        // thread t holds kPer bins from the top, in descending order
        const int b0 = kRadixBins - 1 - kPer * tid;
        int h[kPer], sum = 0;
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
            h[e] = sh.hist[b0 - e];
            sum += h[e];
        }
        int inc = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) sh.scan[warp] = inc;
        __syncthreads();
        int before = lane < warp ? sh.scan[lane] : 0;
        for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xFFFFFFFFu, before, o);
        before += inc - sum;
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
            if (before < need && before + h[e] >= need) {
                sh.digit = b0 - e;
                sh.need = need - before;
            }
            before += h[e];
        }
        __syncthreads();
        prefix |= static_cast<uint32_t>(sh.digit) << shift;
        need = sh.need;
    }
    const int run = ((n + kWarps - 1) / kWarps + 31) / 32 * 32;
    const int r0 = warp * run, r1 = r0 + run < n ? r0 + run : n;
    int gt = 0, eq = 0;
    for (int i = r0 + lane; i < r1; i += 32) {
        const uint32_t key = keys[i];
        gt += key > prefix;
        eq += key == prefix;
    }
    for (int o = 16; o > 0; o >>= 1) {
        gt += __shfl_xor_sync(0xFFFFFFFFu, gt, o);
        eq += __shfl_xor_sync(0xFFFFFFFFu, eq, o);
    }
    if (lane == 0) {
        sh.gt[warp] = gt;
        sh.eq[warp] = eq;
    }
    __syncthreads();
    gt = lane < warp ? sh.gt[lane] : 0;
    eq = lane < warp ? sh.eq[lane] : 0;
    for (int o = 16; o > 0; o >>= 1) {
        gt += __shfl_xor_sync(0xFFFFFFFFu, gt, o);
        eq += __shfl_xor_sync(0xFFFFFFFFu, eq, o);
    }
    const unsigned below = (1u << lane) - 1u;
    for (int i0 = r0; i0 < r1; i0 += 32) {
        const int i = i0 + lane;
        const uint32_t key = i < r1 ? keys[i] : 0u;
        const unsigned bg = __ballot_sync(0xFFFFFFFFu, i < r1 && key > prefix);
        const unsigned be = __ballot_sync(0xFFFFFFFFu, i < r1 && key == prefix);
        const int g_before = gt + __popc(bg & below), e_before = eq + __popc(be & below);
        if ((bg >> lane & 1u) || ((be >> lane & 1u) && e_before < need))
            out[g_before + (e_before < need ? e_before : need)] = static_cast<int32_t>(lo + i);
        gt += __popc(bg);
        eq += __popc(be);
    }
}
constexpr int kTopkUnroll = 16;  // independent loads in flight per thread

// One CTA per unit. Up to kSortMax candidates, topk_emit on the keys in shared
// memory. Beyond that, the
// k-th largest key T is found with four 8-bit radix passes (16 coalesced
// loads in flight per thread); the selected blocks are those with key > T
// plus the lowest-indexed ones with key == T, emitted in ascending block
// order: every warp owns a contiguous segment, counts its picks, and after
// one scan over the warps writes them in order with warp-level prefix sums.
// Both give the same selection.
__global__ void __launch_bounds__(kTopkThreads) k_topk(SelArgs a, const float* __restrict__ scores,
                                                       int32_t* __restrict__ sel,
                                                       int32_t* __restrict__ sel_count)
{
    __shared__ int hist[256];
    __shared__ __align__(16) int whist[kTopkThreads / 32][256];  // per-warp histograms, or keys and scratch
    static_assert(sizeof(whist) >= (kSortMax + kTopkPad) * sizeof(uint32_t) + sizeof(TopkShared), "key buffer");
    __shared__ uint32_t s_prefix;
    __shared__ int s_need;
    const int u_first = unit_lower_bound(a.ut, a.sc_begin);
    const int u_end = unit_lower_bound(a.ut, a.sc_end);
    const int u = u_first + blockIdx.x;
    if (u >= u_end) return;
    int anc;
    int64_t s, e, lo, hi;
    unit_range(a.ut, u, &anc, &s, &e);
    cand_range(a, s, &lo, &hi);
    const int64_t n = hi - lo;
    int32_t* out = sel + static_cast<int64_t>(u) * a.k;
    const float* sc = scores + static_cast<int64_t>(u) * a.nb;

    if (n <= a.k) {
        for (int i = threadIdx.x; i < a.k; i += blockDim.x) out[i] = (i < n) ? static_cast<int32_t>(lo + i) : -1;
        if (threadIdx.x == 0) sel_count[u] = static_cast<int32_t>(n);
        return;
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (a.k == 0) {
        if (threadIdx.x == 0) sel_count[u] = 0;
        return;
    }
    if (n <= kSortMax) {
        uint32_t* sk = reinterpret_cast<uint32_t*>(&whist[0][0]);
        for (int i = threadIdx.x; i < n; i += blockDim.x) sk[i] = float_key(sc[lo + i]);
        __syncthreads();
        topk_emit<kTopkThreads>(sk, static_cast<int>(n), lo, a.k, out, *reinterpret_cast<TopkShared*>(sk + kSortMax + kTopkPad));
        if (threadIdx.x == 0) sel_count[u] = a.k;  // n > k: exactly k picks
        return;
    }
    if (threadIdx.x == 0) {
        s_prefix = 0;
        s_need = a.k;
    }
    uint32_t mask = 0;
    for (int shift = 24; shift >= 0; shift -= 8) {
        for (int i = threadIdx.x; i < (kTopkThreads / 32) * 256; i += blockDim.x) (&whist[0][0])[i] = 0;
        __syncthreads();
        const uint32_t prefix = s_prefix;
        // Every warp counts into its own histogram (keys of similar magnitude
        // share digits, so one shared histogram would serialise on a few bins).
        for (int64_t b0 = lo; b0 < hi; b0 += kTopkUnroll * static_cast<int64_t>(blockDim.x)) {
            uint32_t key[kTopkUnroll];
#pragma unroll
            for (int j = 0; j < kTopkUnroll; ++j) {
                const int64_t b = b0 + j * blockDim.x + threadIdx.x;
                key[j] = b < hi ? float_key(sc[b]) : 0u;
            }
#pragma unroll
            for (int j = 0; j < kTopkUnroll; ++j) {
                const int64_t b = b0 + j * blockDim.x + threadIdx.x;
                const bool in = b < hi && (key[j] & mask) == prefix;
                if (in) atomicAdd(&whist[warp][(key[j] >> shift) & 255u], 1);
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < 256; i += blockDim.x) {
            int c = 0;
            for (int w = 0; w < kTopkThreads / 32; ++w) c += whist[w][i];
            hist[i] = c;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            int need = s_need, cum = 0, d = 255;
            for (; d > 0; --d) {
                if (cum + hist[d] >= need) break;
                cum += hist[d];
            }
            s_need = need - cum;
            s_prefix = prefix | (static_cast<uint32_t>(d) << shift);
        }
        mask |= 255u << shift;
        __syncthreads();
    }
    const uint32_t T = s_prefix;
    const int need_eq = s_need;  // how many keys equal to T to take, lowest b first
    // Ordered compaction: warp w owns the contiguous segment [w0, w1); lane l
    // reads keys w0 + 128 i + 4 l .. + 3, so every step is one coalesced 512-byte
    // read and index order within the warp is (step, lane, j).
    const int nw = blockDim.x >> 5;
    const int64_t seg = ((n + nw - 1) / nw + 127) / 128 * 128;
    const int64_t w0 = lo + seg * warp;
    const int64_t w1 = (w0 + seg < hi) ? w0 + seg : hi;
    auto load4 = [&](int64_t b, uint32_t (&key)[4]) {
#pragma unroll
        for (int j = 0; j < 4; ++j) key[j] = (b + j < w1) ? float_key(sc[b + j]) : 0u;
    };
    int n_gt = 0, n_eq = 0;
    for (int64_t b = w0 + 4 * lane; b < w1; b += 128) {
        uint32_t key[4];
        load4(b, key);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            n_gt += (b + j < w1) && key[j] > T;
            n_eq += (b + j < w1) && key[j] == T;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        n_gt += __shfl_xor_sync(0xFFFFFFFFu, n_gt, o);
        n_eq += __shfl_xor_sync(0xFFFFFFFFu, n_eq, o);
    }
    __shared__ int s_take[kTopkThreads / 32], s_pos[kTopkThreads / 32], s_taken;
    if (lane == 0) {
        s_take[warp] = n_eq;  // equal keys of this warp, for now
        s_pos[warp] = n_gt;   // keys above T of this warp, for now
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int eq_before = 0, pos = 0;
        for (int w = 0; w < nw; ++w) {
            const int e = s_take[w], g = s_pos[w];
            int take = need_eq - eq_before;
            take = take < 0 ? 0 : (take > e ? e : take);
            eq_before += e;
            s_take[w] = take;
            s_pos[w] = pos;
            pos += g + take;
        }
        s_taken = pos;
    }
    __syncthreads();
    const int taken = s_taken;
    int pos = s_pos[warp], take_eq = s_take[warp];
    for (int64_t b = w0 + 4 * lane; b < w1; b += 128) {
        uint32_t key[4];
        load4(b, key);
        int gt_l = 0, eq_l = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            gt_l += (b + j < w1) && key[j] > T;
            eq_l += (b + j < w1) && key[j] == T;
        }
        // exclusive prefix over lanes of the equal keys
        int eq_inc = eq_l;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, eq_inc, o);
            if (lane >= o) eq_inc += y;
        }
        const int eq_tot = __shfl_sync(0xFFFFFFFFu, eq_inc, 31);
        int eq_rank = eq_inc - eq_l;  // equal keys before this lane in this step
        // picks of this lane: keys above T and the equal keys still to take
        int pk[4], n_pk = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            pk[j] = 0;
            if (b + j < w1) {
                if (key[j] > T) pk[j] = 1;
                else if (key[j] == T) pk[j] = (eq_rank++ < take_eq);
            }
            n_pk += pk[j];
        }
        int pk_inc = n_pk;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, pk_inc, o);
            if (lane >= o) pk_inc += y;
        }
        int p = pos + pk_inc - n_pk;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (pk[j]) out[p++] = static_cast<int32_t>(b + j);
        pos += __shfl_sync(0xFFFFFFFFu, pk_inc, 31);
        take_eq -= (eq_tot < take_eq ? eq_tot : take_eq);
    }
    for (int i = taken + threadIdx.x; i < a.k; i += blockDim.x) out[i] = -1;
    if (threadIdx.x == 0) sel_count[u] = taken;
}

// Steps (b)-(c) after the logits for units of at most kSortMax candidates,
// one CTA of kTopkThreads per unit: the heads' statistics, the soft vote
// (scores written where asked for, NaN off the candidates) and the short path
// of k_topk. A warp takes a head's statistics in one pass (each lane the running
// maximum and the sum of exp(z - maximum), so the large terms take no rounding
// of the exponential's argument: raised only by jumps of 8, the errors of rows
// of standard deviation 8 to 12 were up to 9 % larger); both passes over the logits load VEC blocks at a time, which is
// what bounds the kernel: latency times the bytes in flight. 256 units of up to
// 4,096 blocks and 32 heads: 34 us (scalar loads, max and sum in two
// passes: 51 us). VEC is 4 where the rows allow 16-byte loads.
constexpr int kFusedMaxHeads = 256;
template <int VEC>
__global__ void __launch_bounds__(kTopkThreads) k_select_fused(SelArgs a, const float* __restrict__ logits,
                                                               float* __restrict__ scores,
                                                               int32_t* __restrict__ sel,
                                                               int32_t* __restrict__ sel_count)
{
    __shared__ float s_m[kFusedMaxHeads], s_inv[kFusedMaxHeads];
    __shared__ __align__(16) uint32_t sk[kSortMax + kTopkPad];
    __shared__ TopkShared sh;
    scale_ptx::pdl_enter();
    const int u_first = unit_lower_bound(a.ut, a.sc_begin);
    const int u_end = unit_lower_bound(a.ut, a.sc_end);
    const int u = u_first + blockIdx.x;
    if (u >= u_end) return;
    int anc;
    int64_t s, e, lo64, hi64;
    unit_range(a.ut, u, &anc, &s, &e);
    cand_range(a, s, &lo64, &hi64);
    const int lo = static_cast<int>(lo64), hi = static_cast<int>(hi64), n = hi - lo;  // at most kSortMax blocks
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // VEC logits of a row from block b (a multiple of VEC, inside the row)
    auto load = [](const float* z, int b, float (&x)[VEC]) {
        if (VEC == 4) {
            const float4 v = __ldcg(reinterpret_cast<const float4*>(z + b));
            x[0] = v.x;
            x[VEC > 1 ? 1 : 0] = v.y;
            x[VEC > 2 ? 2 : 0] = v.z;
            x[VEC > 3 ? 3 : 0] = v.w;
        } else {
            x[0] = __ldcg(z + b);
        }
    };
    constexpr int kIn = 8;  // loads in flight
    const int first = lo / VEC * VEC;
    const bool rank = n > a.k && a.k > 0;
    if (n > 0 && (rank || scores))
        for (int h = warp; h < a.Hq; h += kTopkThreads / 32) {
            const float* z = logits + (static_cast<int64_t>(u) * a.Hq + h) * a.nb;
            float m = -INFINITY, sum = 0.f;
            for (int b0 = first + VEC * lane; b0 < hi; b0 += 32 * VEC * kIn) {
                float x[kIn][VEC];
#pragma unroll
                for (int i = 0; i < kIn; ++i) {
                    const int b = b0 + 32 * VEC * i;
                    if (b < hi) load(z, b, x[i]);
#pragma unroll
                    for (int c = 0; c < VEC; ++c)
                        if (b + c < lo || b + c >= hi) x[i][c] = -INFINITY;
                }
                float top = x[0][0];
#pragma unroll
                for (int i = 0; i < kIn; ++i)
#pragma unroll
                    for (int c = 0; c < VEC; ++c) top = fmaxf(top, x[i][c]);
                if (top > m) {
                    sum *= exp_factor(m - top);
                    m = top;
                }
                float part = 0.f;
#pragma unroll
                for (int i = 0; i < kIn; ++i)
#pragma unroll
                    for (int c = 0; c < VEC; ++c) part += x[i][c] == -INFINITY ? 0.f : expf(x[i][c] - m);
                sum += part;
            }
            float mm = m;
            for (int o = 16; o > 0; o >>= 1) mm = fmaxf(mm, __shfl_xor_sync(0xFFFFFFFFu, mm, o));
            sum = m == -INFINITY ? 0.f : sum * exp_factor(m - mm);
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
            if (lane == 0) {
                s_m[h] = mm;
                s_inv[h] = 1.0f / sum;
            }
        }
    __syncthreads();
    // soft vote over the heads in order; the candidates' keys
    float* sc = scores ? scores + static_cast<int64_t>(u) * a.nb : nullptr;
    for (int b = VEC * threadIdx.x; b < a.nb; b += VEC * kTopkThreads) {
        float score[VEC];
#pragma unroll
        for (int c = 0; c < VEC; ++c) score[c] = 0.f;
        if (b + VEC > lo && b < hi && (rank || sc)) {
            const float* zb = logits + static_cast<int64_t>(u) * a.Hq * a.nb;
            for (int h0 = 0; h0 < a.Hq; h0 += kIn) {
                float z[kIn][VEC];
#pragma unroll
                for (int i = 0; i < kIn; ++i)
                    load(zb + static_cast<int64_t>(h0 + i < a.Hq ? h0 + i : a.Hq - 1) * a.nb, b, z[i]);
#pragma unroll
                for (int i = 0; i < kIn; ++i)
                    if (h0 + i < a.Hq) {
                        const float mx = s_m[h0 + i], inv = s_inv[h0 + i];
#pragma unroll
                        for (int c = 0; c < VEC; ++c) score[c] += expf(z[i][c] - mx) * inv;
                    }
            }
        }
#pragma unroll
        for (int c = 0; c < VEC; ++c) {
            const bool in = b + c >= lo && b + c < hi;
            if (in && rank) sk[b + c - lo] = float_key(score[c]);
            if (sc) sc[b + c] = in ? score[c] : __int_as_float(0x7FC00000);
        }
    }
    int32_t* out = sel + static_cast<int64_t>(u) * a.k;
    if (!rank) {
        for (int i = threadIdx.x; i < a.k; i += blockDim.x) out[i] = i < n ? lo + i : -1;
        if (threadIdx.x == 0) sel_count[u] = n < a.k ? n : a.k;
        return;
    }
    __syncthreads();
    topk_emit<kTopkThreads>(sk, n, lo, a.k, out, sh);
    if (threadIdx.x == 0) sel_count[u] = a.k;  // n > k: exactly k picks
}

// ---- sequences of little selection work: the whole selection in one launch.

constexpr int kFewRuns = 16;       // runs of a unit's candidates, each with a partial softmax sum
constexpr int kFewThreads = 512;
constexpr int kFewWarps = kFewThreads / 32;
constexpr int kFewSmem = 152 * 1024;
// Values v[0..V) of every lane summed over the 32 lanes: lane c ends with the
// sum of value c % V in v[0] (halving exchanges: V - 1 shuffles, then log2(32 / V)).
template <int V>
__device__ __forceinline__ void reduce_to_lanes(float (&v)[V])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int x = V / 2; x > 0; x >>= 1)
#pragma unroll
        for (int y = 0; y < x; ++y) {
            const float keep = (lane & x) ? v[y + x] : v[y];
            const float give = (lane & x) ? v[y] : v[y + x];
            v[y] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, x);
        }
#pragma unroll
    for (int x = V; x < 32; x <<= 1) v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], x);
}

// A cluster of gridDim.x (1, 2, .. 16) CTAs per unit. The unit's candidate
// blocks are cut into 16 runs, of which every rank owns 16 / gridDim.x
// neighbouring ones. Logits: a warp takes NB blocks of one KV head at a time,
// each lane four of the 128 dimensions of the representatives and of the head's
// G queries, in fp32; they stay in shared memory. Statistics: (max, sum) of
// every run for every head, sent to all ranks. Vote: the runs' (max, sum) merged
// in order, then the scores of the rank's blocks, whose keys go to rank 0, which
// picks the k largest. Nothing but the selection (and the scores, if asked for)
// is written to memory. The arithmetic depends on the unit alone, not on the
// size of the cluster or on the other units of the call: a unit has the same
// scores, bit for bit, in every call. Bound by latency in a large cluster, by
// the shuffles of the dot products and the reads of the representatives from L2
// in a small one (the next item's blocks in flight during them: 1024 x 32 logits
// on one CTA 91 us against 83, not taken); few_ctas chooses by the number of units.
// Dynamic shared memory: logits [H_q][runs of the rank * stride], then keys
// [nb + kTopkPad]. RUNS: runs of a rank, 0 when gridDim.x decides; as a constant
// they save 0.3 us of 5.5 in a cluster of 16.
template <int G, int RUNS>
__global__ void __launch_bounds__(kFewThreads, 1) k_select_few(SelArgs a, const float* __restrict__ fp,
                                                               const float* __restrict__ reps, int stride,
                                                               float* __restrict__ scores,
                                                               int32_t* __restrict__ sel,
                                                               int32_t* __restrict__ sel_count)
{
    using namespace scale_ptx;
    constexpr int NB = G <= 4 ? 8 : 4;
    constexpr int V = G == 1 ? 8 : G == 2 ? 16 : 32;
    extern __shared__ __align__(16) float zs[];  // topk_emit reads the keys behind them 16 bytes at a time
    __shared__ float2 s_part[kFewRuns][kFusedMaxHeads + 1];  // + 1: a head's runs in different banks
    __shared__ float s_m[kFusedMaxHeads], s_inv[kFusedMaxHeads];
    __shared__ TopkShared sh;
    pdl_enter();
    const int u = unit_lower_bound(a.ut, a.sc_begin) + static_cast<int>(blockIdx.y);
    if (u >= unit_lower_bound(a.ut, a.sc_end)) return;  // the whole cluster
    int anc;
    int64_t s, e, lo, hi;
    unit_range(a.ut, u, &anc, &s, &e);
    cand_range(a, s, &lo, &hi);
    const int n = static_cast<int>(hi - lo);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ctas = RUNS ? kFewRuns / RUNS : static_cast<int>(gridDim.x);
    const int runs = RUNS ? RUNS : kFewRuns / ctas;  // of this rank
    const int rank = static_cast<int>(cluster_ctarank());
    float* sc = scores ? scores + static_cast<int64_t>(u) * a.nb : nullptr;
    int32_t* out = sel + static_cast<int64_t>(u) * a.k;
    if (sc)  // NaN off the candidates
        for (int64_t b = rank * kFewThreads + tid; b < a.nb; b += ctas * kFewThreads)
            if (b < lo || b >= hi) sc[b] = __int_as_float(0x7FC00000);
    const bool pick = n > a.k && a.k > 0;
    if (!pick) {  // every candidate, or none
        if (rank == 0) {
            for (int i = tid; i < a.k; i += kFewThreads) out[i] = i < n ? static_cast<int32_t>(lo + i) : -1;
            if (tid == 0) sel_count[u] = n < a.k ? n : a.k;
        }
        if (!sc || n == 0) return;
    }
    cluster_arrive();  // waited for before the first store to another rank: all have started
    const int slice = ((n + kFewRuns - 1) / kFewRuns + NB - 1) / NB * NB;  // blocks of a run, at most `stride`
    const int row = runs * stride;                                         // logits of a head
    const int r0 = rank * runs * slice;
    const int len = n - r0 < runs * slice ? (n - r0 > 0 ? n - r0 : 0) : runs * slice;
    const int Hkv = a.Hq / G;

    // logits of the rank's blocks: items (KV head, NB blocks), a KV head's items on neighbouring warps
    const int nbk = (len + NB - 1) / NB;
    for (int it = warp; it < nbk * Hkv; it += kFewWarps) {
        const int j = it / nbk, b0 = (it - j * nbk) * NB;
        const float4* rp = reinterpret_cast<const float4*>(reps + (j * a.nb + lo + r0 + b0) * kHeadDim) + lane;
        float4 x[NB];
#pragma unroll
        for (int i = 0; i < NB; ++i)
            x[i] = b0 + i < len ? __ldg(rp + i * (kHeadDim / 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4* qp = reinterpret_cast<const float4*>(fp + (static_cast<int64_t>(anc) * a.Hq + j * G) * kHeadDim) + lane;
        float v[V];
#pragma unroll
        for (int i = 0; i < V; ++i) v[i] = 0.f;
#pragma unroll
        for (int hl = 0; hl < G; ++hl) {
            const float4 qv = __ldg(qp + hl * (kHeadDim / 4));
#pragma unroll
            for (int i = 0; i < NB; ++i)
                v[hl * NB + i] = fmaf(qv.x, x[i].x, qv.y * x[i].y) + fmaf(qv.z, x[i].z, qv.w * x[i].w);
        }
        reduce_to_lanes<V>(v);
        if (lane < G * NB) zs[(j * G + lane / NB) * row + b0 + lane % NB] = a.sigma * v[0];
    }
    cluster_wait();
    __syncthreads();
    // (max, sum) of every run per head, to every rank (lane r to rank r); a warp
    // takes heads h and h + half of a run at a time, their chains side by side
    const int half = (a.Hq + 1) / 2;
    for (int x = warp; x < runs * half; x += kFewWarps) {
        const int run = runs == 1 ? 0 : x / half, h0 = x - run * half;
        const int cnt = len - run * slice < slice ? len - run * slice : slice;
        float m[2] = {-INFINITY, -INFINITY}, sum[2] = {0.f, 0.f};
        const float* zh[2] = {zs + h0 * row + run * slice, zs + (h0 + half < a.Hq ? h0 + half : h0) * row + run * slice};
        for (int i = lane; i < cnt; i += 32)
#pragma unroll
            for (int c = 0; c < 2; ++c) m[c] = fmaxf(m[c], zh[c][i]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int c = 0; c < 2; ++c) m[c] = fmaxf(m[c], __shfl_xor_sync(0xFFFFFFFFu, m[c], o));
        for (int i = lane; i < cnt; i += 32)
#pragma unroll
            for (int c = 0; c < 2; ++c) sum[c] += expf(zh[c][i] - m[c]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int c = 0; c < 2; ++c) sum[c] += __shfl_xor_sync(0xFFFFFFFFu, sum[c], o);
#pragma unroll
        for (int c = 0; c < 2; ++c)
            if (lane < ctas && h0 + c * half < a.Hq)
                st_cluster_f2(cluster_map(&s_part[rank * runs + run][h0 + c * half], lane), m[c], sum[c]);
    }
    cluster_arrive();
    cluster_wait();
    static_assert(kFewRuns == 16, "half a warp merges the runs of a head");
    for (int x = tid; x - tid < a.Hq * kFewRuns; x += kFewThreads) {
        const int h = x / kFewRuns;
        const float2 part = h < a.Hq ? s_part[x % kFewRuns][h] : make_float2(-INFINITY, 0.f);
        float m = part.x;
#pragma unroll
        for (int o = kFewRuns / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
        float sum = part.x > -INFINITY ? part.y * exp_factor(part.x - m) : 0.f;
#pragma unroll
        for (int o = kFewRuns / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
        if (h < a.Hq && x % kFewRuns == 0) {
            s_m[h] = m;
            s_inv[h] = 1.0f / sum;
        }
    }
    __syncthreads();
    uint32_t* keys = reinterpret_cast<uint32_t*>(zs + static_cast<size_t>(a.Hq) * row);
    const uint32_t keys0 = cluster_map(keys, 0);
    for (int i = tid; i < len; i += kFewThreads) {
        float score = 0.f;
        for (int h = 0; h < a.Hq; ++h) score += expf(zs[h * row + i] - s_m[h]) * s_inv[h];
        if (sc) sc[lo + r0 + i] = score;
        if (pick) st_cluster_u32(keys0 + 4 * (r0 + i), float_key(score));
    }
    cluster_arrive();  // after it rank 0 has every key and no rank's shared memory is written
    cluster_wait();
    if (rank != 0 || !pick) return;
    topk_emit<kFewThreads>(keys, n, lo, a.k, out, sh);
    if (tid == 0) sel_count[u] = a.k;
}

// Blocks of a run in shared memory, and the bytes of a rank in clusters of
// `ctas` (0 when they do not fit).
int few_stride(const Derived& d)
{
    return static_cast<int>(((d.nb + kFewRuns - 1) / kFewRuns + 7) / 8 * 8);
}
size_t few_smem(const Derived& d, int ctas)
{
    const int64_t bytes = (static_cast<int64_t>(few_stride(d)) * (kFewRuns / ctas) * d.Hq + d.nb + kTopkPad) * 4;
    return bytes <= kFewSmem ? static_cast<size_t>(bytes) : 0;
}

// Time of one SM for a unit's candidates, in ns: the dot products and votes grow
// with the query heads, the reads of the representatives with the KV heads.
int64_t few_work(const Derived& d) { return d.nb * (d.Hq + 4 * d.Hkv); }

// Whether the sequence's selection runs in k_select_few, whatever the range of a
// call: the scores of k_logits and k_select_fused differ from its in the last
// bits, and a unit must have the same scores, and so the same blocks, in a call
// of its own and in one over the whole sequence. k_select_few is faster in
// calls of few units (the loop over outer chunks), the other kernels over many;
// GPU time per call, 32 heads on 8, one unit and 64 units:
//   blocks              256          512         1024         2048         4096
//   k_select_few     9.4  20.5   9.8  28.5   12.4  45.6   17.0  80.0   26.5  146 us
//   the others      16.6  17.3  17.4  18.4   18.3  21.7   21.6  29.5   35.7   50 us
// The line is where a call over the whole sequence takes about twice as long
// (64 units of 1024 blocks); the kernels beyond kSortMax blocks are slower (8192
// blocks: one unit 84 us against 45, 64 units 115 against 215, 256 units 252
// against 809 us beside a layer's attention of some 100 ms).
constexpr int64_t kFewLine = 1ll << 22;
constexpr int64_t kFewLineLong = 1ll << 27;
bool few_sequence(const Derived& d)
{
    return d.g <= 8 && d.Hq <= kFusedMaxHeads && few_smem(d, kFewRuns) > 0 &&
           d.M * few_work(d) <= (d.nb <= kSortMax ? kFewLine : kFewLineLong);
}

// CTAs of a unit's cluster: the size with the shortest call by estimate, the
// rounds of the clusters that run at once times 5 us and the unit's work.
// Measured, 32 heads on 8 and 256 / 1024 blocks, clusters of 16, 8, 4, 2, 1:
//    1 unit    9.4 / 12.3   10.5 / 16.6   13.8 / 25.9   20.4 / 44.8   33.2 / 82.7 us
//   14 units  14.8 / 21.3   10.6 / 17.0   13.8 / 26.3   20.3 / 45.1   33.0 / 82.1
//   36 units  35.0 / 54.7   23.6 / 41.9   14.0 / 26.6   20.4 / 45.3   33.2 / 82.3
//   64 units  55.6 / 86.6   36.6 / 65.3   26.1 / 50.0   20.6 / 45.6   33.1 / 82.2
int few_ctas(const Derived& d, int units)
{
    constexpr int kSlots[5] = {7, 14, 36, 76, 152};  // clusters of 16, 8, 4, 2, 1 at once
    int best = 0;
    float least = 0.f;
    for (int i = 0; i < 5; ++i) {
        const int ctas = kFewRuns >> i;
        if (!few_smem(d, ctas)) break;
        const float us = static_cast<float>((units + kSlots[i] - 1) / kSlots[i]) *
                         (5.0f + 1e-3f * static_cast<float>(few_work(d)) / static_cast<float>(ctas));
        if (!best || us < least) {
            best = ctas;
            least = us;
        }
    }
    return best;
}

// Units to expect among `max_units` sub-chunks: the host does not know the
// clusters that a threshold has closed, between one per S_max sub-chunks and one
// each; the geometric mean of the two is off by no more than sqrt(S_max) either way.
int few_units(const Derived& d, bool per_subchunk, int max_units)
{
    if (per_subchunk) return max_units;
    const int per_outer = d.per_outer < max_units ? d.per_outer : max_units;
    const int size = d.S_max < per_outer ? d.S_max : per_outer;
    const float least = std::ceil(static_cast<float>(max_units) / static_cast<float>(size));
    return static_cast<int>(d.theta <= -1.0f ? least : std::ceil(std::sqrt(least * static_cast<float>(max_units))));
}

template <int G>
cudaError_t run_select_few(const Derived& d, const SelArgs& a, int ctas, int max_units, const float* fp,
                           const float* reps, float* scores, int32_t* sel, int32_t* sel_count, cudaStream_t st)
{
    auto kern = ctas == kFewRuns ? k_select_few<G, 1> : k_select_few<G, 0>;
    // set on every launch: the attributes belong to the current device
    const size_t smem = few_smem(d, ctas);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e == cudaSuccess && ctas == kFewRuns)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    return launch_after(st, dim3(static_cast<unsigned>(ctas), static_cast<unsigned>(max_units)), kFewThreads, smem,
                        ctas, kern, a, fp, reps, few_stride(d), scores, sel, sel_count);
}

cudaError_t launch_select_few(const Derived& d, const SelArgs& a, int ctas, int max_units, const float* fp,
                              const float* reps, float* scores, int32_t* sel, int32_t* sel_count, cudaStream_t st)
{
    switch (d.g) {
    case 1: return run_select_few<1>(d, a, ctas, max_units, fp, reps, scores, sel, sel_count, st);
    case 2: return run_select_few<2>(d, a, ctas, max_units, fp, reps, scores, sel, sel_count, st);
    case 3: return run_select_few<3>(d, a, ctas, max_units, fp, reps, scores, sel, sel_count, st);
    case 4: return run_select_few<4>(d, a, ctas, max_units, fp, reps, scores, sel, sel_count, st);
    case 5: return run_select_few<5>(d, a, ctas, max_units, fp, reps, scores, sel, sel_count, st);
    case 6: return run_select_few<6>(d, a, ctas, max_units, fp, reps, scores, sel, sel_count, st);
    case 7: return run_select_few<7>(d, a, ctas, max_units, fp, reps, scores, sel, sel_count, st);
    default: return run_select_few<8>(d, a, ctas, max_units, fp, reps, scores, sel, sel_count, st);
    }
}

// ---- top-k over many candidates per unit: the same radix select and ordered
// output as k_topk, spread over CTAs of kChunk candidates (grid y = unit).

constexpr int kChunk = 2048;              // candidates per CTA and pass
constexpr int64_t kMultiCtaMin = 65536;   // more candidates than this: the multi-CTA form
constexpr int kChunkThreads = 256;

struct TopkState {
    uint32_t prefix;  // bits of the k-th key fixed so far
    int need;         // keys still to take at or below the prefix
    int done;         // 1: the unit's output is already complete
    int pad;
};
static_assert(sizeof(TopkState) == 4 * sizeof(int32_t), "TopkState is four int32 words");

__device__ __forceinline__ bool unit_cands(const SelArgs& a, int ui, int* u, int64_t* lo, int64_t* hi)
{
    const int u_first = unit_lower_bound(a.ut, a.sc_begin);
    const int u_end = unit_lower_bound(a.ut, a.sc_end);
    *u = u_first + ui;
    if (*u >= u_end) return false;
    int anc;
    int64_t s, e;
    unit_range(a.ut, *u, &anc, &s, &e);
    cand_range(a, s, lo, hi);
    return true;
}

// Per unit: small candidate sets are written out directly; otherwise the
// radix state starts (prefix 0, need k) and the four passes' histograms are
// cleared. state[u][i] is the state after the digits of i passes are fixed;
// the kernel that first needs state i + 1 derives it from state i and the
// histogram of pass i (its CTA 0 stores it for the kernels after it).
__global__ void __launch_bounds__(256) k_topk_init(SelArgs a, int32_t* __restrict__ sel,
                                                    int32_t* __restrict__ sel_count, int32_t* __restrict__ hist,
                                                    TopkState* __restrict__ state)
{
    int u;
    int64_t lo, hi;
    if (!unit_cands(a, blockIdx.x, &u, &lo, &hi)) return;
    const int64_t n = hi - lo;
    for (int i = threadIdx.x; i < kTopkPasses * 256; i += blockDim.x) hist[u * kTopkPasses * 256 + i] = 0;
    if (n <= a.k) {
        int32_t* out = sel + static_cast<int64_t>(u) * a.k;
        for (int i = threadIdx.x; i < a.k; i += blockDim.x) out[i] = (i < n) ? static_cast<int32_t>(lo + i) : -1;
        if (threadIdx.x == 0) {
            sel_count[u] = static_cast<int32_t>(n);
            state[u * (kTopkPasses + 1)] = TopkState{0u, 0, 1, 0};
        }
    } else if (threadIdx.x == 0) {
        state[u * (kTopkPasses + 1)] = TopkState{0u, a.k, 0, 0};
    }
}

// State after pass p (p >= 1): the digit of the k-th largest key at the
// shift of pass p - 1, from that pass's histogram and the state before it
// (the largest digit d whose keys, with those above it, reach `need`).
// Every thread of the CTA returns it; CTA 0 stores it.
__device__ TopkState topk_state_after(const int32_t* __restrict__ hist_u, TopkState* __restrict__ state_u,
                                      int p, bool store)
{
    __shared__ int h[256];
    __shared__ TopkState s_st;
    for (int i = threadIdx.x; i < 256; i += blockDim.x) h[i] = hist_u[(p - 1) * 256 + i];
    __syncthreads();
    if (threadIdx.x == 0) {
        TopkState stt = state_u[p - 1];
        int need = stt.need, cum = 0, d = 255;
        for (; d > 0; --d) {
            if (cum + h[d] >= need) break;
            cum += h[d];
        }
        stt.need = need - cum;
        stt.prefix |= static_cast<uint32_t>(d) << (24 - 8 * (p - 1));
        s_st = stt;
        if (store) state_u[p] = stt;
    }
    __syncthreads();
    return s_st;
}

// Radix pass p (shift 24 - 8 p): per-warp histograms of the digit at `shift`
// of the keys that match the prefix fixed by the passes before, added into
// the unit's histogram of pass p.
__global__ void __launch_bounds__(kChunkThreads) k_topk_hist(SelArgs a, const float* __restrict__ scores,
                                                             int32_t* __restrict__ hist,
                                                             TopkState* __restrict__ state, int p)
{
    __shared__ int wh[kChunkThreads / 32][256];
    int u;
    int64_t lo, hi;
    if (!unit_cands(a, blockIdx.y, &u, &lo, &hi)) return;
    TopkState* su = state + u * (kTopkPasses + 1);
    int32_t* hu = hist + u * kTopkPasses * 256;
    if (su[0].done) return;
    const int64_t c0 = lo + static_cast<int64_t>(blockIdx.x) * kChunk;
    if (c0 >= hi) return;
    const int shift = 24 - 8 * p;
    const TopkState stt = p == 0 ? su[0] : topk_state_after(hu, su, p, blockIdx.x == 0);
    const int64_t c1 = (c0 + kChunk < hi) ? c0 + kChunk : hi;
    const int warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < (kChunkThreads / 32) * 256; i += blockDim.x) (&wh[0][0])[i] = 0;
    __syncthreads();
    const uint32_t mask = shift == 24 ? 0u : (0xFFFFFFFFu << (shift + 8));
    const float* sc = scores + static_cast<int64_t>(u) * a.nb;
    constexpr int kPer = kChunk / kChunkThreads;
    uint32_t key[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int64_t b = c0 + j * kChunkThreads + threadIdx.x;
        key[j] = b < c1 ? float_key(sc[b]) : 0u;
    }
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int64_t b = c0 + j * kChunkThreads + threadIdx.x;
        if (b < c1 && (key[j] & mask) == stt.prefix) atomicAdd(&wh[warp][(key[j] >> shift) & 255u], 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 256; i += blockDim.x) {
        int c = 0;
        for (int w = 0; w < kChunkThreads / 32; ++w) c += wh[w][i];
        if (c) atomicAdd(&hu[p * 256 + i], c);
    }
}

// Counts per chunk of the keys above the k-th key T and of the keys equal to it.
// The k-th key T is the prefix after the last pass (derived here, stored by CTA 0).
__global__ void __launch_bounds__(kChunkThreads) k_topk_count(SelArgs a, const float* __restrict__ scores,
                                                              const int32_t* __restrict__ hist,
                                                              TopkState* __restrict__ state,
                                                              int2* __restrict__ counts, int max_chunks)
{
    int u;
    int64_t lo, hi;
    if (!unit_cands(a, blockIdx.y, &u, &lo, &hi)) return;
    TopkState* su = state + u * (kTopkPasses + 1);
    if (su[0].done) return;
    const int64_t c0 = lo + static_cast<int64_t>(blockIdx.x) * kChunk;
    if (c0 >= hi) return;
    const TopkState stt = topk_state_after(hist + u * kTopkPasses * 256, su, kTopkPasses, blockIdx.x == 0);
    const int64_t c1 = (c0 + kChunk < hi) ? c0 + kChunk : hi;
    const float* sc = scores + static_cast<int64_t>(u) * a.nb;
    int gt = 0, eq = 0;
    for (int64_t b = c0 + threadIdx.x; b < c1; b += blockDim.x) {
        const uint32_t key = float_key(sc[b]);
        gt += key > stt.prefix;
        eq += key == stt.prefix;
    }
    for (int o = 16; o > 0; o >>= 1) {
        gt += __shfl_xor_sync(0xFFFFFFFFu, gt, o);
        eq += __shfl_xor_sync(0xFFFFFFFFu, eq, o);
    }
    __shared__ int sg[kChunkThreads / 32], se[kChunkThreads / 32];
    if ((threadIdx.x & 31) == 0) {
        sg[threadIdx.x >> 5] = gt;
        se[threadIdx.x >> 5] = eq;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int g = 0, e = 0;
        for (int w = 0; w < kChunkThreads / 32; ++w) {
            g += sg[w];
            e += se[w];
        }
        counts[static_cast<int64_t>(u) * max_chunks + blockIdx.x] = make_int2(g, e);
    }
}

// Per unit: output position and number of equal keys to take of every chunk
// (the equal keys are taken lowest index first); the -1 padding and the count.
__global__ void __launch_bounds__(32) k_topk_scan(SelArgs a, const TopkState* __restrict__ state,
                                                   int2* __restrict__ counts, int max_chunks,
                                                   int32_t* __restrict__ sel, int32_t* __restrict__ sel_count)
{
    int u;
    int64_t lo, hi;
    if (!unit_cands(a, blockIdx.x, &u, &lo, &hi)) return;
    if (state[u * (kTopkPasses + 1)].done) return;
    const TopkState stt = state[u * (kTopkPasses + 1) + kTopkPasses];
    const int n_chunks = static_cast<int>((hi - lo + kChunk - 1) / kChunk);
    int2* cu = counts + static_cast<int64_t>(u) * max_chunks;
    // Two prefix sums over the chunks, 32 at a time with the totals carried:
    // the equal keys before each chunk (how many of its equal keys it takes
    // follows), then the picks before it (its output position).
    const int lane = threadIdx.x;
    int eq_run = 0, pos_run = 0;
    for (int c0 = 0; c0 < n_chunks; c0 += 32) {
        const int c = c0 + lane;
        const int2 ge = c < n_chunks ? cu[c] : make_int2(0, 0);
        int eq_inc = ge.y;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, eq_inc, o);
            if (lane >= o) eq_inc += y;
        }
        const int eq_before = eq_run + eq_inc - ge.y;
        int take = stt.need - eq_before;
        take = take < 0 ? 0 : (take > ge.y ? ge.y : take);
        const int picks = ge.x + take;
        int pos_inc = picks;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, pos_inc, o);
            if (lane >= o) pos_inc += y;
        }
        if (c < n_chunks) cu[c] = make_int2(pos_run + pos_inc - picks, take);
        eq_run += __shfl_sync(0xFFFFFFFFu, eq_inc, 31);
        pos_run += __shfl_sync(0xFFFFFFFFu, pos_inc, 31);
    }
    if (lane == 0) sel_count[u] = pos_run;
    int32_t* out = sel + static_cast<int64_t>(u) * a.k;
    for (int i = pos_run + lane; i < a.k; i += 32) out[i] = -1;
}

// Ordered output of one chunk: every warp owns a contiguous segment (lane l
// reads 4 consecutive keys per step), counts its picks, and after a scan over
// the warps writes them in index order with warp prefix sums.
__global__ void __launch_bounds__(kChunkThreads) k_topk_emit(SelArgs a, const float* __restrict__ scores,
                                                             const TopkState* __restrict__ state,
                                                             const int2* __restrict__ counts, int max_chunks,
                                                             int32_t* __restrict__ sel)
{
    int u;
    int64_t lo, hi;
    if (!unit_cands(a, blockIdx.y, &u, &lo, &hi)) return;
    if (state[u * (kTopkPasses + 1)].done) return;
    const TopkState stt = state[u * (kTopkPasses + 1) + kTopkPasses];
    const int64_t c0 = lo + static_cast<int64_t>(blockIdx.x) * kChunk;
    if (c0 >= hi) return;
    const int64_t c1 = (c0 + kChunk < hi) ? c0 + kChunk : hi;
    const int2 pt = counts[static_cast<int64_t>(u) * max_chunks + blockIdx.x];
    const uint32_t T = stt.prefix;
    const float* sc = scores + static_cast<int64_t>(u) * a.nb;
    int32_t* out = sel + static_cast<int64_t>(u) * a.k;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int nw = kChunkThreads / 32;
    const int64_t seg = kChunk / nw;
    const int64_t w0 = c0 + seg * warp;
    const int64_t w1 = (w0 + seg < c1) ? w0 + seg : c1;
    int n_gt = 0, n_eq = 0;
    for (int64_t b = w0 + 4 * lane; b < w1; b += 128)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (b + j < w1) {
                const uint32_t key = float_key(sc[b + j]);
                n_gt += key > T;
                n_eq += key == T;
            }
    for (int o = 16; o > 0; o >>= 1) {
        n_gt += __shfl_xor_sync(0xFFFFFFFFu, n_gt, o);
        n_eq += __shfl_xor_sync(0xFFFFFFFFu, n_eq, o);
    }
    __shared__ int s_take[nw], s_pos[nw];
    if (lane == 0) {
        s_take[warp] = n_eq;
        s_pos[warp] = n_gt;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int eq_before = 0, pos = pt.x;
        for (int w = 0; w < nw; ++w) {
            const int e = s_take[w], g = s_pos[w];
            int take = pt.y - eq_before;
            take = take < 0 ? 0 : (take > e ? e : take);
            eq_before += e;
            s_take[w] = take;
            s_pos[w] = pos;
            pos += g + take;
        }
    }
    __syncthreads();
    int pos = s_pos[warp], take_eq = s_take[warp];
    for (int64_t b = w0 + 4 * lane; b < w1; b += 128) {
        uint32_t key[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) key[j] = (b + j < w1) ? float_key(sc[b + j]) : 0u;
        int eq_l = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) eq_l += (b + j < w1) && key[j] == T;
        int eq_inc = eq_l;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, eq_inc, o);
            if (lane >= o) eq_inc += y;
        }
        const int eq_tot = __shfl_sync(0xFFFFFFFFu, eq_inc, 31);
        int eq_rank = eq_inc - eq_l;
        int pk[4], n_pk = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            pk[j] = 0;
            if (b + j < w1) {
                if (key[j] > T) pk[j] = 1;
                else if (key[j] == T) pk[j] = (eq_rank++ < take_eq);
            }
            n_pk += pk[j];
        }
        int pk_inc = n_pk;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xFFFFFFFFu, pk_inc, o);
            if (lane >= o) pk_inc += y;
        }
        int p = pos + pk_inc - n_pk;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (pk[j]) out[p++] = static_cast<int32_t>(b + j);
        pos += __shfl_sync(0xFFFFFFFFu, pk_inc, 31);
        take_eq -= (eq_tot < take_eq ? eq_tot : take_eq);
    }
}

}  // namespace

int topk_max_chunks(const Derived& d) { return static_cast<int>((d.nb + kChunk - 1) / kChunk); }

cudaError_t launch_select(const Derived& d, int mode, int64_t tok_begin, int64_t tok_end,
                          const float* reps, const float* fingerprints, const int32_t* unit_start,
                          const int32_t* n_units, int32_t* sel_blocks, int32_t* sel_count,
                          float* sel_scores, uint8_t* ws, uint64_t timeout_ns, cudaStream_t st)
{
    const WsLayout lay = ws_layout(d);
    float* logits = reinterpret_cast<float*>(ws + lay.logits);
    float* stats = reinterpret_cast<float*>(ws + lay.stats);
    float* scores = sel_scores ? sel_scores : reinterpret_cast<float*>(ws + lay.scores);

    SelArgs a{};
    a.ut = Units{unit_start, n_units, mode == SCALE_MODE_PER_SUBCHUNK, d.N, d.L, static_cast<int>(d.M)};
    a.sc_begin = static_cast<int>(tok_begin / d.L);
    a.sc_end = static_cast<int>((tok_end + d.L - 1) / d.L);
    a.Hq = d.Hq;
    a.g = d.g;
    a.nb = d.nb;
    a.B = d.B;
    a.k = d.k;
    a.n_sink = d.n_sink;
    a.n_local = d.n_local;
    a.sigma = d.sigma;
    a.scored = sel_scores != nullptr;
    a.status = reinterpret_cast<int32_t*>(ws + kStatusOffset);
    a.timeout_ns = timeout_ns;
    const int max_units = a.sc_end - a.sc_begin;  // units in range <= sub-chunks in range
    if (max_units <= 0) return cudaSuccess;

    if (few_sequence(d)) {
        // A large cluster may not be had everywhere (a partition of the device);
        // nothing is enqueued then and a smaller one does the same work, or the
        // kernels below where its share does not fit.
        for (int ctas = few_ctas(d, few_units(d, a.ut.per_subchunk, max_units)); ctas && few_smem(d, ctas); ctas /= 2) {
            const cudaError_t ef = launch_select_few(d, a, ctas, max_units, fingerprints, reps, sel_scores, sel_blocks,
                                                     sel_count, st);
            if (ef == cudaSuccess) return ef;
            cudaGetLastError();
        }
    }
    // Tiles per CTA: as many as leave every SM a CTA, at most kLtSeg.
    int sms = 0;
    cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    const int upt = kLtRows / d.g;  // units per logits tile
    const int tiles = (max_units + upt - 1) / upt;
    const int64_t ctas = static_cast<int64_t>(tiles) * ((d.nb + 127) / 128) * d.Hkv;
    const int seg = ctas >= static_cast<int64_t>(kLtSeg) * sms ? kLtSeg : static_cast<int>((ctas + sms - 1) / sms);
    // set on every launch: the attribute belongs to the current device
    e = cudaFuncSetAttribute(k_logits, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kLtSmem));
    if (e != cudaSuccess) return e;
    dim3 gl((tiles + seg - 1) / seg, static_cast<unsigned>((d.nb + 127) / 128), d.Hkv);
    e = launch_after(st, gl, kLtThreads, kLtSmem, 1, k_logits, a, seg, fingerprints, reps, logits);
    if (e != cudaSuccess) return e;
    if (d.nb <= kSortMax && d.Hq <= kFusedMaxHeads && d.k <= kSortMax) {
        // every unit's candidates fit the sort: statistics, vote and top-k in one kernel
        return launch_after(st, dim3(max_units), kTopkThreads, 0, 1,
                            d.nb % 4 == 0 ? k_select_fused<4> : k_select_fused<1>, a, logits, sel_scores, sel_blocks,
                            sel_count);
    }
    const int64_t rows = static_cast<int64_t>(max_units) * d.Hq;
    k_stats<<<static_cast<unsigned>((rows + 7) / 8), 256, 0, st>>>(a, logits, stats);
    k_vote<<<dim3(static_cast<unsigned>((d.nb + 255) / 256), max_units), 256, 0, st>>>(a, logits, stats, scores);
    k_topk<<<max_units, kTopkThreads, 0, st>>>(a, scores, sel_blocks, sel_count);
    return cudaGetLastError();
}

cudaError_t launch_topk(const Derived& d, const Units& ut, int sc_begin, int sc_end, const float* scores,
                        int32_t* sel, int32_t* sel_count, cudaStream_t st, const TopkScratch& scratch)
{
    SelArgs a{};
    a.ut = ut;
    a.sc_begin = sc_begin;
    a.sc_end = sc_end;
    a.Hq = d.Hq;
    a.g = d.g;
    a.nb = d.nb;
    a.B = d.B;
    a.k = d.k;
    a.n_sink = d.n_sink;
    a.n_local = d.n_local;
    a.sigma = d.sigma;
    const int max_units = sc_end - sc_begin;
    if (max_units <= 0) return cudaSuccess;
    if (d.nb <= kMultiCtaMin) {
        k_topk<<<max_units, kTopkThreads, 0, st>>>(a, scores, sel, sel_count);
        return cudaGetLastError();
    }
    // many candidates per unit: chunks of kChunk keys over the whole GPU
    auto* state = reinterpret_cast<TopkState*>(scratch.state);
    const int mc = scratch.max_chunks;
    const dim3 grid(static_cast<unsigned>(mc), static_cast<unsigned>(max_units));
    k_topk_init<<<max_units, 256, 0, st>>>(a, sel, sel_count, scratch.hist, state);
    for (int p = 0; p < kTopkPasses; ++p)
        k_topk_hist<<<grid, kChunkThreads, 0, st>>>(a, scores, scratch.hist, state, p);
    k_topk_count<<<grid, kChunkThreads, 0, st>>>(a, scores, scratch.hist, state, scratch.counts, mc);
    k_topk_scan<<<max_units, 32, 0, st>>>(a, state, scratch.counts, mc, sel, sel_count);
    k_topk_emit<<<grid, kChunkThreads, 0, st>>>(a, scores, state, scratch.counts, mc, sel);
    return cudaGetLastError();
}

}  // namespace scale
