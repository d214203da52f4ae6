// score.cu -- selection at block size 1 for few units (every call of the
// Algorithm 2 loop, and a decode step): the soft-vote scores and the top-k
// from one read of K, in two kernels.
//
//   k_key_logits  z[u][h][t] = v_u^(h) . k_t^(h/g) for the candidate tokens,
//                 written to a plane in the workspace, and per CTA the
//                 (reference, sum) of each head's softmax;
//   k_vote_topk   one cooperative launch: the heads' statistics, the soft vote
//                 score[u][t] = sum_h 2^(z scale2 - m_h) / s_h, and the k
//                 largest scores (ties to the lower token, ascending output).
//
// One read of K plus a plane of 4 H_q bytes per (unit, token), written and
// read once, replaces two reads of K (512 H_kv bytes per token each): 256
// against 2,048 bytes per token and unit for 32 query heads on 8 KV heads.
#include <cuda_bf16.h>

#include <type_traits>

#include "launch.cuh"
#include "ptx_sm103.cuh"
#include "scale_internal.h"
#include "score.cuh"
#include "tma_host.h"

namespace scale {
namespace {

using namespace scale_ptx;

// ---------------------------------------------------------------- logits

constexpr int kLgThreads = 192;
constexpr int kLgStages = 3;
constexpr int64_t kLgStreamBytes = 64ll << 20;  // keys: half of L2
constexpr int64_t kLgShareBytes = 88ll << 20;   // keys: two thirds of L2
constexpr int64_t kLgPlaneBytes = 96ll << 20;   // planes: what L2 still holds beside them
constexpr int kLgFold = 16;                     // key tiles summed before they join a column's total
constexpr int kLgCols = 16;                     // (unit, head) columns of a tile
constexpr uint32_t kLgTile = 128 * 128 * 2;     // 128 keys x 128 dims, two 64-dim halves
constexpr uint32_t kLgHalf = kLgTile / 2;
constexpr float kFar = 1073741824.0f;           // 2^30: references whose neighbours are 64 apart
constexpr uint32_t kLgOpMax = 3 * kLgCols * 256;  // query operand: up to 48 rows of 256 bytes
constexpr uint32_t kLgSmem = kLgOpMax + kLgStages * kLgTile + 1024;
static_assert(kLgOpMax % 1024 == 0, "key stages must stay 1024-aligned");
static_assert(2 * (kLgSmem + 2048) <= 227 * 1024, "two CTAs per SM");

struct LgBars {
    uint64_t f_full, f_empty;
    uint64_t k_full[kLgStages], k_empty[kLgStages];
    uint64_t d_full[2], d_empty[2];
    uint64_t drain;
};

__device__ __forceinline__ void lg_fail(volatile int* abort_flag, int32_t* status)
{
    *abort_flag = 1;
    record_status(status, SCALE_ERR_TIMEOUT);
}

__device__ __forceinline__ int64_t unit_window(const Units& ut, int n_local, int u)
{
    int anc;
    int64_t s, e;
    unit_range(ut, u, &anc, &s, &e);
    return s - n_local > 0 ? s - n_local : 0;
}

// The CTAs [part_first, part_end) of k_key_logits can have items of KV head j.
__device__ __forceinline__ int part_first(int j, int n_part, int Hkv)
{
    return static_cast<int>(static_cast<int64_t>(j) * n_part / Hkv);
}
__device__ __forceinline__ int part_end(int j, int n_part, int Hkv)
{
    return static_cast<int>((static_cast<int64_t>(j + 1) * n_part + Hkv - 1) / Hkv);
}

// Whether a decode step retrieves (Eq. 8 across steps): no when the cosine of
// its query with the cached anchor reaches theta and the anchor's selection
// still may be shared. Every CTA computes it with the same arithmetic in the
// same order, so all decide alike without a launch of its own; the state and
// the anchor are updated by the attention kernel of the step. All threads call.
__device__ bool decode_retrieves(const KeyScoreArgs& a)
{
    __shared__ float red[3][kLgThreads / 32];
    const int D8 = a.Hq * kHeadDim / 8;
    const uint4* q = reinterpret_cast<const uint4*>(a.q);
    const float4* an = reinterpret_cast<const float4*>(a.anchor);
    float dot = 0.f, nq = 0.f, na = 0.f;
    constexpr int kIn = 3;  // 32 heads: every load of the thread in flight
    for (int i0 = threadIdx.x; i0 < D8; i0 += kIn * kLgThreads) {
        uint4 x[kIn];
        float4 y0[kIn], y1[kIn];
#pragma unroll
        for (int b = 0; b < kIn; ++b) {
            const int i = i0 + b * kLgThreads < D8 ? i0 + b * kLgThreads : i0;
            x[b] = q[i];
            y0[b] = an[2 * i];
            y1[b] = an[2 * i + 1];
        }
#pragma unroll
        for (int b = 0; b < kIn; ++b) {
            if (i0 + b * kLgThreads >= D8) continue;
            const uint32_t w[4] = {x[b].x, x[b].y, x[b].z, x[b].w};
            const float y[8] = {y0[b].x, y0[b].y, y0[b].z, y0[b].w, y1[b].x, y1[b].y, y1[b].z, y1[b].w};
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const float v = __uint_as_float(c & 1 ? w[c / 2] & 0xFFFF0000u : w[c / 2] << 16);
                dot += v * y[c];
                nq += v * v;
                na += y[c] * y[c];
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        dot += __shfl_xor_sync(0xFFFFFFFFu, dot, o);
        nq += __shfl_xor_sync(0xFFFFFFFFu, nq, o);
        na += __shfl_xor_sync(0xFFFFFFFFu, na, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = dot;
        red[1][threadIdx.x >> 5] = nq;
        red[2][threadIdx.x >> 5] = na;
    }
    __syncthreads();
    float d = 0.f, a2 = 0.f, b2 = 0.f;
    for (int i = 0; i < kLgThreads / 32; ++i) {
        d += red[0][i];
        a2 += red[1][i];
        b2 += red[2][i];
    }
    const float cs = (a2 > 0.f && b2 > 0.f) ? d / (sqrtf(a2) * sqrtf(b2)) : 0.f;  // zero norm: 0
    return !(a.state[0] && a.state[1] < a.S_max && cs >= a.theta);
}

// Grid (n_part CTAs, unit tiles of 16 / G units). The work of a unit tile is
// its items (KV head j, 128-token key tile), head by head, cut into n_part
// equal runs, one per CTA, so every CTA streams one long run of a head's keys
// whatever the length of the sequence, and two CTAs per SM keep up to six
// 32 KB tiles in flight. Warp 0 lane 0 issues the TMA loads (the query operand
// when the head changes, the key tiles into a 3-stage ring), warp 1 lane 0 the
// MMAs (rows = the tile's 128 tokens, columns = PARTS x 16: the bf16 parts of
// the 16 (unit, head) columns side by side; a decode query is bf16 itself, one
// part), warps 2-5 add the parts, write z and keep each column's running
// (max, sum) in the token's thread, merged over the 128 threads (a butterfly,
// then the four warps in order) when the head changes. Bound by reading K,
// with many unit tiles by the planes. The CTAs of the unit tiles that read the
// same keys run side by side when L2 does not hold all keys: selection calls of
// 16 units of 32 heads take 107 us at 48K tokens, 208 at 128K and 896 at 512K
// (tile after tile 121, 256 and 1018); where L2 holds them the order matters
// little (40K tokens: 98.2 side by side, 100.6 tile after tile, which is taken).
template <int G, int PARTS>
__global__ void __launch_bounds__(kLgThreads, 2)
k_key_logits(const __grid_constant__ CUtensorMap tf, const __grid_constant__ CUtensorMap tk, const KeyScoreArgs a)
{
    constexpr int US = kLgCols / G;               // units of the tile
    constexpr int NC = PARTS == 1 ? G : kLgCols;  // columns read back
    constexpr uint32_t kOpHalf = PARTS * kLgCols * 128;
    constexpr uint32_t kAcc = PARTS == 1 ? 16 : 64;  // TMEM columns of an accumulator
    extern __shared__ uint8_t smem_raw[];
    __shared__ LgBars bars;
    __shared__ uint32_t tmem_slot;
    __shared__ volatile int abort_flag;
    __shared__ int s_W[US];
    __shared__ float s_max[4][kLgCols], s_sum[4][kLgCols];
    pdl_enter();

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int u_first = unit_lower_bound(a.ut, a.sc_begin);
    const int u_end = unit_lower_bound(a.ut, a.sc_end);
    if (u_first >= u_end) return;
    const int u_tiles = (u_end - u_first + US - 1) / US;  // at most gridDim.y
    int cta = blockIdx.x, ut = blockIdx.y;                // run of the items, unit tile
    // Keys beyond what L2 holds: the unit tiles take the same keys at the same time
    if (PARTS > 1 && u_tiles > 1 &&
        unit_window(a.ut, a.n_local, u_end - 1) * a.Hkv * (kHeadDim * 2) > kLgShareBytes) {
        const int linear = static_cast<int>(blockIdx.y * gridDim.x + blockIdx.x);
        cta = linear / u_tiles;
        ut = linear % u_tiles;
    }
    if (ut >= u_tiles || cta >= static_cast<int>(gridDim.x)) return;
    const int ui0 = ut * US;  // first unit of the tile, from the range's first
    const int u0 = u_first + ui0;
    const int n_u = (u_end - u0 < US) ? u_end - u0 : US;

    // k_vote_topk finds its histograms and counters cleared
    for (int ul = 0; ul < n_u; ++ul) {
        int32_t* sc = a.scratch + static_cast<int64_t>(ui0 + ul) * kVoteScratchInts;
        for (int i = cta * kLgThreads + tid; i < kVoteCounts; i += gridDim.x * kLgThreads) sc[i] = 0;
    }
    if (PARTS == 1) {
        for (int i = tid; i < a.Hkv && cta == 0; i += kLgThreads) a.tickets[i] = 0;
        const bool retrieve = decode_retrieves(a);
        if (cta == 0 && tid == 0) *a.gate = retrieve;
        if (!retrieve) return;
    }

    const int64_t w_max = unit_window(a.ut, a.n_local, u0 + n_u - 1);
    const int hi = static_cast<int>(w_max < a.N ? w_max : a.N);
    const int lo = a.n_sink / 128 * 128;  // key tiles start at a multiple of 128: inside one KV page
    const int64_t tiles = hi > a.n_sink ? (hi - lo + 127) / 128 : 0;
    const int64_t items = tiles * a.Hkv;
    const int64_t i0 = items * cta / gridDim.x, i1 = items * (cta + 1) / gridDim.x;
    const int n_it = static_cast<int>(i1 - i0);
    const int j_first = n_it ? static_cast<int>(i0 / tiles) : 0;
    const int j_last = n_it ? static_cast<int>((i1 - 1) / tiles) : -1;
    // heads that k_vote_topk looks for in this CTA although it has no item of them
    for (int x = tid; x < n_u * a.Hq; x += kLgThreads) {
        const int j = x % a.Hq / G;
        if ((j < j_first || j > j_last) && cta >= part_first(j, a.n_part, a.Hkv) &&
            cta < part_end(j, a.n_part, a.Hkv))
            a.part[(static_cast<int64_t>(ui0) * a.Hq + x) * a.n_part + cta] = make_float2(-INFINITY, 0.f);
    }
    if (n_it == 0) return;
    const int t_first = static_cast<int>(i0 - j_first * tiles);  // tile of the first item

    uint8_t* smem = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
    uint8_t* kbuf = smem + kLgOpMax;
    if (tid < US) s_W[tid] = (tid < n_u) ? static_cast<int>(unit_window(a.ut, a.n_local, u0 + tid)) : 0;
    if (tid == 0) {
        abort_flag = 0;
        mbar_init(&bars.f_full, 1);
        mbar_init(&bars.f_empty, 1);
        for (int i = 0; i < kLgStages; ++i) {
            mbar_init(&bars.k_full[i], 1);
            mbar_init(&bars.k_empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&bars.d_full[i], 1);
            mbar_init(&bars.d_empty[i], 128);
        }
        mbar_init(&bars.drain, 1);
        fence_barrier_init();
    }
    if (warp == 1) {
        tmem_alloc(&tmem_slot, 2 * kAcc);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp == 0) {
        // ------------------------------------------------------------ producer
        if (lane == 0) {
            tma_prefetch_desc(&tf);
            tma_prefetch_desc(&tk);
            // Keys beyond what L2 holds leave it before the planes that the vote
            // reads, as long as L2 holds those: a decode step of 32 heads takes
            // 84.7 us at 128K tokens and 223.2 at 512K (a plane of 64 MB), 92.1
            // and 229.3 without. Planes larger than L2 are read from HBM all the
            // same, and the policy only costs: 416.9 us at 1M, 412.5 without; a
            // selection of 16 units at 256K tokens 477 and 381.
            const int64_t plane = items * 128 * G * 4 * (u_end - u_first);
            const bool stream = items * static_cast<int64_t>(kLgTile) > kLgStreamBytes && plane <= kLgPlaneBytes;
            const uint64_t policy = policy_evict_first();
            int issued = 0, issued_f = 0;
            int j = j_first - 1, tile = static_cast<int>(tiles), st = 0, ph = 1;
            for (int it = 0; it < n_it && !abort_flag; ++it) {
                if (it == 0 || ++tile == tiles) {  // the next head's query operand
                    tile = it == 0 ? t_first : 0;
                    ++j;
                    if (issued_f && !mbar_wait_bounded(&bars.f_empty, (issued_f - 1) & 1, a.timeout_ns, &abort_flag)) {
                        lg_fail(&abort_flag, a.status);
                        break;
                    }
                    mbar_arrive_expect_tx(&bars.f_full, 2 * kOpHalf);
                    ++issued_f;
                    for (int sp = 0; sp < PARTS; ++sp)
                        for (int hf = 0; hf < 2; ++hf)
                            tma_load_4d(smem + hf * kOpHalf + sp * kLgCols * 128, &tf, &bars.f_full, hf * 64,
                                        PARTS == 1 ? j * G : u0 * G, PARTS == 1 ? 0 : j, sp);
                }
                if (it >= kLgStages && !mbar_wait_bounded(&bars.k_empty[st], ph, a.timeout_ns, &abort_flag)) {
                    lg_fail(&abort_flag, a.status);
                    break;
                }
                mbar_arrive_expect_tx(&bars.k_full[st], kLgTile);
                ++issued;
                const int32_t ra = kv_row_tma(a.pg, lo + 128ll * tile);
                const int32_t rb = kv_row_tma(a.pg, lo + 128ll * tile + 64);
                for (int hf = 0; hf < 2; ++hf) {
                    uint8_t* dst = kbuf + st * kLgTile + hf * kLgHalf;
                    if (stream) {
                        tma_load_3d_hint(dst, &tk, &bars.k_full[st], hf * 64, j, ra, policy);
                        tma_load_3d_hint(dst + kLgHalf / 2, &tk, &bars.k_full[st], hf * 64, j, rb, policy);
                    } else {
                        tma_load_3d(dst, &tk, &bars.k_full[st], hf * 64, j, ra);
                        tma_load_3d(dst + kLgHalf / 2, &tk, &bars.k_full[st], hf * 64, j, rb);
                    }
                }
                if (++st == kLgStages) {
                    st = 0;
                    ph ^= 1;
                }
            }
            if (abort_flag) {
                if (issued_f) mbar_wait_bounded(&bars.f_full, (issued_f - 1) & 1, a.timeout_ns, nullptr);
                for (int i = 0; i < kLgStages; ++i) {
                    const int n_i = (issued + kLgStages - 1 - i) / kLgStages;  // copies into stage i
                    if (n_i) mbar_wait_bounded(&bars.k_full[i], (n_i - 1) & 1, a.timeout_ns, nullptr);
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            const uint32_t idesc = idesc_bf16_f32(128, PARTS * kLgCols, 0);
            const uint64_t fdesc = sdesc_sw128(smem_addr(smem), 16, 1024);
            const uint64_t kdesc0 = sdesc_sw128(smem_addr(kbuf), 16, 1024);
            bool ok = true;
            int tile = 0, heads = 0, st = 0, ph = 0;
            for (int it = 0; it < n_it; ++it) {
                if (it == 0 || ++tile == tiles) {
                    if (it > 0) mma_commit(&bars.f_empty);
                    tile = it == 0 ? t_first : 0;
                    if (!mbar_wait_bounded(&bars.f_full, heads & 1, a.timeout_ns, &abort_flag)) { ok = false; break; }
                    ++heads;
                }
                const int b = it & 1;
                if (!mbar_wait_bounded(&bars.k_full[st], ph, a.timeout_ns, &abort_flag)) { ok = false; break; }
                if (it >= 2 && !mbar_wait_bounded(&bars.d_empty[b], ((it >> 1) - 1) & 1, a.timeout_ns, &abort_flag)) { ok = false; break; }
                tc_fence_after();
                mma_ss_k128_ab<kLgHalf, kOpHalf>(tmem + b * kAcc, kdesc0 + st * (kLgTile >> 4), fdesc, idesc, 0u);
                mma_commit(&bars.d_full[b]);
                mma_commit(&bars.k_empty[st]);
                if (++st == kLgStages) {
                    st = 0;
                    ph ^= 1;
                }
            }
            if (!ok) {
                lg_fail(&abort_flag, a.status);
                mma_commit(&bars.drain);
                mbar_wait_bounded(&bars.drain, 0, a.timeout_ns, nullptr);
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue
        // The four warps see the same heads, so their named barriers match,
        // also after a failed wait (the work is then skipped).
        const int q = warp & 3;  // TMEM lane quarter this warp may access
        const int r = q * 32 + lane;
        const uint32_t lane_base = tmem + (static_cast<uint32_t>(q * 32) << 16);
        bool ok = true;
        int j = j_first, tile = t_first;
        // per column: reference, the sum of the last few tiles, and of those before
        // them (two levels keep the rounding of a run of hundreds of tiles small)
        float m[NC], sm[NC], tot[NC];
        int fresh = 0;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            m[c] = -INFINITY;
            sm[c] = tot[c] = 0.f;
        }
        for (int it = 0; it < n_it; ++it) {
            const int b = it & 1;
            if (ok)
                ok = __all_sync(0xFFFFFFFFu,
                                mbar_wait_bounded(&bars.d_full[b], (it >> 1) & 1, a.timeout_ns, &abort_flag));
            if (ok) {
                tc_fence_after();
                float z[NC];
                if (PARTS == 1) {
                    uint32_t p0[16];
                    tmem_ld16(lane_base + b * kAcc, p0);
                    tmem_ld_wait();
#pragma unroll
                    for (int c = 0; c < NC; ++c) z[c] = __uint_as_float(p0[c]);
                } else {
                    uint32_t p0[16], p1[16], p2[16];
                    tmem_ld16(lane_base + b * kAcc, p0);
                    tmem_ld16(lane_base + b * kAcc + kLgCols, p1);
                    tmem_ld16(lane_base + b * kAcc + 2 * kLgCols, p2);
                    tmem_ld_wait();
#pragma unroll
                    for (int c = 0; c < NC; ++c)
                        z[c] = (__uint_as_float(p0[c]) + __uint_as_float(p1[c])) + __uint_as_float(p2[c]);
                }
                tc_fence_before();
                mbar_arrive(&bars.d_empty[b]);
                const int t0 = lo + 128 * tile, t = t0 + r;
                float* zt = a.z + (static_cast<int64_t>(ui0) * a.Hq + j * G) * a.z_stride + t;
                // The reference m is a whole number, so that every factor between
                // references is an exact power of two, and z scale2 - m is rounded
                // once, by the size of the difference. (With the product rounded
                // first and references raised by jumps of 2^8, the scores of logits of
                // standard deviation 3 were 31e-8 from 64 bits at 100,003 tokens; now
                // 10e-8.) Beyond kFar the rounding of the product alone is larger than
                // the exponential's range: a thread's sum then counts as 1, at the end.
                // The raise stays as short as this: one instruction more, and the
                // compiler no longer predicates it, which costs 12 %.
                auto raise = [&](int c, float& x) {
                    const float top = ceilf(z[c] * a.scale2), f = ex2(m[c] - top);
                    sm[c] *= f;
                    tot[c] *= f;
                    m[c] = top;
                    x = fminf(fmaf(z[c], a.scale2, -top), 1.0f);
                };
                // A tile of candidates of every unit (the windows ascend) goes through
                // its units without a test per value, and looks for a larger reference
                // once: 8 units at 300K tokens, 28 heads on 4, 222 us (a test per value
                // 260), one unit at 1M, 32 on 8, 375 us (386).
                if (t0 >= a.n_sink && t0 + 127 < s_W[0]) {
                    float x[US * G], most = -INFINITY;
#pragma unroll
                    for (int ul = 0; ul < US; ++ul) {
                        if (ul >= n_u) break;
#pragma unroll
                        for (int c = ul * G; c < (ul + 1) * G && c < NC; ++c) {
                            zt[(static_cast<int64_t>(ul) * a.Hq + c % G) * a.z_stride] = z[c];
                            x[c] = fmaf(z[c], a.scale2, -m[c]);
                            most = fmaxf(most, x[c]);
                        }
                    }
                    if (most > 0.0f) {
#pragma unroll
                        for (int c = 0; c < US * G && c < NC; ++c)
                            if (c / G < n_u && x[c] > 0.0f) raise(c, x[c]);
                    }
#pragma unroll
                    for (int ul = 0; ul < US; ++ul) {
                        if (ul >= n_u) break;
#pragma unroll
                        for (int c = ul * G; c < (ul + 1) * G && c < NC; ++c) sm[c] += ex2(x[c]);
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const int ul = c / G, hl = c % G;
                        if (ul < n_u && t >= a.n_sink && t < s_W[ul < US ? ul : 0]) {
                            zt[(static_cast<int64_t>(ul) * a.Hq + hl) * a.z_stride] = z[c];
                            float x = fmaf(z[c], a.scale2, -m[c]);
                            if (x > 0.0f) raise(c, x);
                            sm[c] += ex2(x);
                        }
                    }
                }
                if (++fresh == kLgFold) {
                    fresh = 0;
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        tot[c] += sm[c];
                        sm[c] = 0.f;
                    }
                }
            }
            if (++tile == tiles || it + 1 == n_it) {
                // The CTA's share of KV head j is complete: one reference for its 128
                // threads (the lanes', then the warps' largest), to which each
                // scales its sums once; lanes added as a tree, warps in order.
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    tot[c] += sm[c];
                    if (fabsf(m[c]) >= kFar && m[c] > -INFINITY) tot[c] = 1.0f;
                    sm[c] = m[c];  // from here on this thread's own reference
                    for (int o = 16; o > 0; o >>= 1) m[c] = fmaxf(m[c], __shfl_xor_sync(0xFFFFFFFFu, m[c], o));
                    if (lane == 0) s_max[q][c] = m[c];
                }
                named_barrier(1, 128);
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const float mm = fmaxf(fmaxf(s_max[0][c], s_max[1][c]), fmaxf(s_max[2][c], s_max[3][c]));
                    float t = sm[c] == -INFINITY ? 0.f : tot[c] * ex2(sm[c] - mm);
                    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, o);
                    if (lane == 0) s_sum[q][c] = t;
                    m[c] = -INFINITY;
                    sm[c] = tot[c] = 0.f;
                }
                fresh = 0;
                named_barrier(1, 128);
                if (r < NC && r / G < n_u && ok)
                    a.part[(static_cast<int64_t>(ui0 + r / G) * a.Hq + j * G + r % G) * a.n_part + cta] =
                        make_float2(fmaxf(fmaxf(s_max[0][r], s_max[1][r]), fmaxf(s_max[2][r], s_max[3][r])),
                                    ((s_sum[0][r] + s_sum[1][r]) + s_sum[2][r]) + s_sum[3][r]);
                named_barrier(1, 128);
                tile = 0;
                ++j;
            }
        }
        if (!ok) lg_fail(&abort_flag, a.status);
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 2 * kAcc);
    }
}

// ---------------------------------------------------------------- vote and top-k

constexpr int kVtThreads = 512;
constexpr int kVtWarps = kVtThreads / 32;
constexpr int kVtBinsPer = kVoteBins / kVtThreads;  // histogram bins of a thread
constexpr int kVtMaxHeads = 512;  // 64 KV heads of at most 8 query heads
constexpr int kVtCopies = 4;       // histogram copies: warps of equal warp % 4 share one
constexpr int kVtKeys = 32768;     // keys of a CTA kept in shared memory
constexpr uint32_t kVtSmem = kVtKeys * 4;

// Order-preserving map of a float onto uint32 (larger float -> larger key).
__device__ __forceinline__ uint32_t float_key(float f)
{
    const uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Inclusive sum over the block in thread order. `sh`: kVtWarps ints; called by all threads.
__device__ __forceinline__ int block_inclusive(int v, int* sh)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xFFFFFFFFu, v, o);
        if (lane >= o) v += y;
    }
    __syncthreads();
    if (lane == 31) sh[warp] = v;
    __syncthreads();
    int before = lane < warp ? sh[lane] : 0;
    for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xFFFFFFFFu, before, o);
    return v + before;
}

// Barrier number `round` (from 1) of the `per` CTAs that work on one unit:
// `counter` was zero before the launch, and the launch is cooperative, so all
// of them are resident. Bounded; false when the wait ran out.
__device__ bool group_barrier(int32_t* counter, int target, uint64_t timeout_ns, int32_t* status)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(counter, 1);
        int ok = 1;
        const uint64_t t0 = globaltimer_ns();
        for (uint32_t it = 1;; ++it) {
            int v;
            asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
            if (v >= target) break;
            if ((it & 63u) == 0u && globaltimer_ns() - t0 > timeout_ns) {
                ok = 0;
                record_status(status, SCALE_ERR_TIMEOUT);
                break;
            }
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// One CTA per SM; the CTAs are shared out evenly over the units of the call,
// each taking a contiguous slice of its unit's candidates, whose keys stay in
// shared memory (slices beyond kVtKeys tokens in the first row of the z plane).
// Statistics: every CTA merges the heads' partials for itself. Then the vote,
// and a radix select of the k-th largest key T in digits of 11, 11 and 10
// bits: the CTA's histogram (in shared memory) is added into the unit's, and
// after a barrier every CTA reads off the digit. The picks are the keys above
// T and the first `need` equal to it; the CTAs' counts are exchanged at the
// last barrier, and each CTA writes its picks in token order. Bound by reading
// the plane and, below some 100K tokens, by its four barriers of about 2 us.
// Measured for one unit with 32 heads: 50 us at 1M tokens (20 us of HBM time)
// and 23 us at 128K, against 142 and about 60 us for the statistics, the vote
// and the eight top-k launches it replaces.
__global__ void __launch_bounds__(kVtThreads, 1) k_vote_topk(const VoteArgs a)
{
    extern __shared__ uint32_t s_keys[];
    __shared__ int s_hist[kVtCopies][kVoteBins];
    __shared__ float2 s_stat[kVtMaxHeads];
    __shared__ int s_scan[kVtWarps], s_gt[kVtWarps], s_eq[kVtWarps];
    __shared__ int s_digit, s_need, s_far;
    pdl_trigger();  // launched plainly: what is before it has completed
    if (a.gate && !*a.gate) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int u_first = unit_lower_bound(a.ut, a.sc_begin);
    const int n_u = unit_lower_bound(a.ut, a.sc_end) - u_first;
    if (n_u <= 0) return;
    const int groups = n_u < static_cast<int>(gridDim.x) ? n_u : static_cast<int>(gridDim.x);
    const int per = gridDim.x / groups;
    const int cid = blockIdx.x % per;
    if (static_cast<int>(blockIdx.x) / per >= groups) return;

    for (int ui = blockIdx.x / per; ui < n_u; ui += groups) {
        const int u = u_first + ui;
        const int row = a.single ? 0 : u;
        const int64_t W = unit_window(a.ut, a.n_local, u);
        const int lo = a.n_sink;
        const int hi = static_cast<int>(W < a.N ? W : a.N);
        const int n = hi > lo ? hi - lo : 0;
        float* z = a.z + static_cast<int64_t>(ui) * a.Hq * a.z_stride;
        float* scores = a.scores ? a.scores + static_cast<int64_t>(u) * a.N : nullptr;
        int32_t* out = a.sel + static_cast<int64_t>(row) * a.k;
        int32_t* scratch = a.scratch + static_cast<int64_t>(ui) * kVoteScratchInts;
        int32_t* counter = scratch + kVoteCounter;
        int2* counts = reinterpret_cast<int2*>(scratch + kVoteCounts);
        // slices start at multiples of four tokens: 16-byte loads of the planes
        const int base = lo & ~3;
        const int slice = ((hi > base ? hi - base : 0) + per - 1) / per + 3 & ~3;
        const int64_t c0 = base + static_cast<int64_t>(cid) * slice;
        const int v0 = c0 < lo ? lo - static_cast<int>(c0) : 0;  // candidates of the slice: c0 + [v0, v1)
        const int v1 = c0 < hi ? static_cast<int>(hi - c0 < slice ? hi - c0 : slice) : 0;
        uint32_t* keys = slice <= kVtKeys ? s_keys : reinterpret_cast<uint32_t*>(z + c0);

        if (scores)  // NaN off the candidates
            for (int64_t t = static_cast<int64_t>(cid) * kVtThreads + tid; t < a.N; t += static_cast<int64_t>(per) * kVtThreads)
                if (t < lo || t >= hi) scores[t] = __int_as_float(0x7FC00000);
        const bool rank = n > a.k && a.k > 0;
        if (!rank) {  // every candidate, or none
            for (int i = cid * kVtThreads + tid; i < a.k; i += per * kVtThreads) out[i] = i < n ? lo + i : -1;
            if (cid == 0 && tid == 0) a.sel_count[row] = n < a.k ? n : a.k;
            if (!scores || n == 0) continue;
        }
        // statistics: one warp per head; the parts in a fixed interleave and tree
        if (tid == 0) s_far = 0;
        __syncthreads();
        for (int h = warp; h < a.Hq; h += kVtWarps) {
            const float2* pr = a.part + (static_cast<int64_t>(ui) * a.Hq + h) * a.n_part;
            float m = -INFINITY, s = 0.f;
            const int x0 = part_first(h / a.g, a.n_part, a.Hq / a.g) + lane, x1 = part_end(h / a.g, a.n_part, a.Hq / a.g);
            for (int x = x0; x < x1; x += 32) m = fmaxf(m, pr[x].x);
            for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
            for (int x = x0; x < x1; x += 32)
                if (pr[x].x > -INFINITY) s += pr[x].y * ex2(pr[x].x - m);
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
            if (lane == 0) {
                s_stat[h] = make_float2(m, s > 0.f ? 1.0f / s : 0.f);
                if (fabsf(m) >= kFar) s_far = 1;
            }
        }
        for (int i = tid; i < kVtCopies * kVoteBins; i += kVtThreads) (&s_hist[0][0])[i] = 0;
        __syncthreads();
        // the vote: four tokens per thread, the loads of kVoteGroup planes in
        // flight, added as a tree, the groups in order; `far`: with the product
        // rounded first, as the reference's was, so that its token keeps its weight
        auto vote = [&](auto far) {
            for (int i = 4 * tid; i < v1; i += 4 * kVtThreads) {
                const float* zt = z + c0 + i;
                float sc[4] = {0.f, 0.f, 0.f, 0.f};
                for (int h0 = 0; h0 < a.Hq; h0 += kVoteGroup) {
                    float4 x[kVoteGroup];
#pragma unroll
                    for (int e = 0; e < kVoteGroup; ++e)
                        if (h0 + e < a.Hq)
                            x[e] = __ldcg(reinterpret_cast<const float4*>(zt + static_cast<int64_t>(h0 + e) * a.z_stride));
#pragma unroll
                    for (int e = 0; e < kVoteGroup; ++e) {
                        const float2 st = h0 + e < a.Hq ? s_stat[h0 + e] : make_float2(INFINITY, 0.f);
                        if (h0 + e >= a.Hq) x[e] = make_float4(0.f, 0.f, 0.f, 0.f);
                        auto weight = [&](float v) {
                            return ex2(decltype(far)::value ? __fmul_rn(v, a.scale2) - st.x : fmaf(v, a.scale2, -st.x)) * st.y;
                        };
                        x[e] = make_float4(weight(x[e].x), weight(x[e].y), weight(x[e].z), weight(x[e].w));
                    }
#pragma unroll
                    for (int w = kVoteGroup / 2; w > 0; w >>= 1)
#pragma unroll
                        for (int e = 0; e < w; ++e) {
                            x[e].x += x[e + w].x;
                            x[e].y += x[e + w].y;
                            x[e].z += x[e + w].z;
                            x[e].w += x[e + w].w;
                        }
                    sc[0] += x[0].x;
                    sc[1] += x[0].y;
                    sc[2] += x[0].z;
                    sc[3] += x[0].w;
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (i + e < v0 || i + e >= v1) continue;
                    if (scores) scores[c0 + i + e] = sc[e];
                    if (rank) {
                        const uint32_t key = float_key(sc[e]);
                        keys[i + e] = key;
                        atomicAdd(&s_hist[warp % kVtCopies][key >> 21], 1);
                    }
                }
            }
        };
        if (s_far) vote(std::true_type{});
        else vote(std::false_type{});
        if (!rank) continue;

        uint32_t prefix = 0;
        int need = a.k;
        for (int p = 0; p < 3; ++p) {
            const int shift = p == 0 ? 21 : p == 1 ? 10 : 0;
            __syncthreads();
            for (int b = tid; b < kVoteBins; b += kVtThreads) {
                int c = 0;
#pragma unroll
                for (int x = 0; x < kVtCopies; ++x) {
                    c += s_hist[x][b];
                    s_hist[x][b] = 0;
                }
                if (c) atomicAdd(&scratch[p * kVoteBins + b], c);
            }
            if (!group_barrier(counter, (p + 1) * per, a.timeout_ns, a.status)) return;
            // the largest digit whose keys, with those above it, reach `need`:
            // thread t holds kVtBinsPer bins from the top, in descending order
            const int b0 = kVoteBins - 1 - kVtBinsPer * tid;
            int h[kVtBinsPer], sum = 0;
#pragma unroll
            for (int e = 0; e < kVtBinsPer; ++e) {
                h[e] = __ldcg(&scratch[p * kVoteBins + b0 - e]);
                sum += h[e];
            }
            int before = block_inclusive(sum, s_scan) - sum;
#pragma unroll
            for (int e = 0; e < kVtBinsPer; ++e) {
                if (before < need && before + h[e] >= need) {
                    s_digit = b0 - e;
                    s_need = need - before;
                }
                before += h[e];
            }
            __syncthreads();
            prefix |= static_cast<uint32_t>(s_digit) << shift;
            need = s_need;
            if (p < 2) {
                const int next = p == 0 ? 10 : 0;
                const uint32_t mask = (1u << (p == 0 ? 11 : 10)) - 1u;
                for (int i = v0 + tid; i < v1; i += kVtThreads) {
                    const uint32_t key = keys[i];
                    if ((key >> shift) == (prefix >> shift))
                        atomicAdd(&s_hist[warp % kVtCopies][(key >> next) & mask], 1);
                }
            }
        }
        // T = prefix; every warp owns a contiguous run of the slice
        const int run = ((v1 - v0 + kVtWarps - 1) / kVtWarps + 31) / 32 * 32;
        const int r0 = v0 + warp * run, r1 = r0 + run < v1 ? r0 + run : v1;
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
            s_gt[warp] = gt;
            s_eq[warp] = eq;
        }
        __syncthreads();
        int wg = lane < warp ? s_gt[lane] : 0, we = lane < warp ? s_eq[lane] : 0;
        int tg = lane < kVtWarps ? s_gt[lane] : 0, te = lane < kVtWarps ? s_eq[lane] : 0;
        for (int o = 16; o > 0; o >>= 1) {
            wg += __shfl_xor_sync(0xFFFFFFFFu, wg, o);
            we += __shfl_xor_sync(0xFFFFFFFFu, we, o);
            tg += __shfl_xor_sync(0xFFFFFFFFu, tg, o);
            te += __shfl_xor_sync(0xFFFFFFFFu, te, o);
        }
        if (tid == 0) __stcg(&counts[cid], make_int2(tg, te));
        if (!group_barrier(counter, 4 * per, a.timeout_ns, a.status)) return;
        // picks of the CTAs before this one (every warp adds them for itself)
        gt = eq = 0;
#pragma unroll
        for (int e = 0; e < kVoteMaxCtas / 32; ++e)
            if (lane + 32 * e < cid) {
                const int2 ge = __ldcg(&counts[lane + 32 * e]);
                gt += ge.x;
                eq += ge.y;
            }
        for (int o = 16; o > 0; o >>= 1) {
            gt += __shfl_xor_sync(0xFFFFFFFFu, gt, o);
            eq += __shfl_xor_sync(0xFFFFFFFFu, eq, o);
        }
        gt += wg;
        eq += we;
        const unsigned below = (1u << lane) - 1u;
        for (int i0 = r0; i0 < r1; i0 += 32) {
            const int i = i0 + lane;
            const uint32_t key = i < r1 ? keys[i] : 0u;
            const unsigned bg = __ballot_sync(0xFFFFFFFFu, i < r1 && key > prefix);
            const unsigned be = __ballot_sync(0xFFFFFFFFu, i < r1 && key == prefix);
            const int g_before = gt + __popc(bg & below), e_before = eq + __popc(be & below);
            if ((bg >> lane & 1u) || ((be >> lane & 1u) && e_before < need))
                out[g_before + (e_before < need ? e_before : need)] = static_cast<int32_t>(c0 + i);
            gt += __popc(bg);
            eq += __popc(be);
        }
        if (cid == 0 && tid == 0) a.sel_count[row] = a.k;  // n > k: exactly k picks
        __syncthreads();
    }
}

template <int G, int PARTS>
cudaError_t run_key_logits(const CUtensorMap& tf, const CUtensorMap& tk, const KeyScoreArgs& a, int max_units,
                           cudaStream_t st)
{
    // set on every launch: the attribute belongs to the current device
    cudaError_t e = cudaFuncSetAttribute(k_key_logits<G, PARTS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(kLgSmem));
    if (e != cudaSuccess) return e;
    constexpr int US = kLgCols / G;
    const dim3 grid(static_cast<unsigned>(a.n_part), static_cast<unsigned>((max_units + US - 1) / US));
    return launch_after(st, grid, kLgThreads, kLgSmem, 1, k_key_logits<G, PARTS>, tf, tk, a);
}

template <int PARTS>
cudaError_t run_key_logits(int g, const CUtensorMap& tf, const CUtensorMap& tk, const KeyScoreArgs& a,
                           int max_units, cudaStream_t st)
{
    switch (g) {
    case 1: return run_key_logits<1, PARTS>(tf, tk, a, max_units, st);
    case 2: return run_key_logits<2, PARTS>(tf, tk, a, max_units, st);
    case 3: return run_key_logits<3, PARTS>(tf, tk, a, max_units, st);
    case 4: return run_key_logits<4, PARTS>(tf, tk, a, max_units, st);
    case 5: return run_key_logits<5, PARTS>(tf, tk, a, max_units, st);
    case 6: return run_key_logits<6, PARTS>(tf, tk, a, max_units, st);
    case 7: return run_key_logits<7, PARTS>(tf, tk, a, max_units, st);
    case 8: return run_key_logits<8, PARTS>(tf, tk, a, max_units, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t device_sms(int* sms)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
    return e;
}

int key_logits_parts(int64_t cand_end, int Hkv, int64_t room)
{
    int sms = 0;
    if (device_sms(&sms) != cudaSuccess) return 0;
    const int64_t items = (cand_end + 127) / 128 * Hkv;
    int64_t n = 2ll * sms;
    if (n > items) n = items;
    if (n > room) n = room;
    return static_cast<int>(n > 0 ? n : 1);
}

cudaError_t launch_key_logits(const KeyScoreArgs& a, int g, bool decode, const void* operand, int64_t M,
                              const void* k, int max_units, cudaStream_t st)
{
    CUtensorMap tf, tk;
    const uint64_t fdims[4] = {kHeadDim, static_cast<uint64_t>(decode ? a.Hq : M * g),
                               static_cast<uint64_t>(decode ? 1 : a.Hkv), decode ? 1u : 3u};
    const uint32_t fbox[4] = {64, kLgCols, 1, 1};
    if (!scale_host::make_dense_bf16_map(&tf, operand, 4, fdims, fbox) ||
        !scale_host::make_token_major_map(&tk, k, kHeadDim, a.Hkv, a.pg.page_table ? a.pg.pool_rows : a.pg.N, 64, 64))
        return cudaErrorInvalidValue;
    return decode ? run_key_logits<1>(g, tf, tk, a, max_units, st) : run_key_logits<3>(g, tf, tk, a, max_units, st);
}

cudaError_t launch_vote_topk(const VoteArgs& a, cudaStream_t st)
{
    int sms = 0;
    cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_vote_topk, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kVtSmem));
    if (e != cudaSuccess) return e;
    VoteArgs args = a;
    void* params[] = {&args};
    // Cooperative: the CTAs wait for one another. Where fewer SMs than the
    // device has are to be had (a partition of it), fewer CTAs do the work.
    for (int grid = sms < kVoteMaxCtas ? sms : kVoteMaxCtas;; grid /= 2) {
        e = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k_vote_topk), dim3(static_cast<unsigned>(grid)),
                                        dim3(kVtThreads), params, kVtSmem, st);
        if (e != cudaSuccess) cudaGetLastError();  // reported by the return value
        if (e != cudaErrorCooperativeLaunchTooLarge || grid == 1) return e;
    }
}

}  // namespace scale
