// decode.cu -- one decode step with a selection cache.
//
// The paper's method targets prefill and leaves decode to the underlying
// engine, whose selection cache reuses a token selection across consecutive,
// highly similar decode queries (Sec. VII, TPOT). This file implements that
// step with the paper's own rules at C = 1 (Def. 1: a decode step processes
// one token):
//  - selection (Eq. 9 at block size 1): the query q_t of position t is the
//    unit's fingerprint; candidates n_sink <= c < W_t, W_t = max(0, t -
//    n_local); per-head softmax over the candidates, head soft-vote, top-k
//    tokens (ties to the lower index), ascending;
//  - cache (Eq. 8 / Algorithm 1 across steps): the query of the last step that
//    retrieved is the anchor; a step reuses the anchor's selection while
//    cos(q_t, anchor) >= theta and fewer than max_cluster_subchunks steps
//    have shared it, and retrieves (and becomes the anchor) otherwise;
//  - attention (Eq. 10 for one row): keys = sinks U selection U [W_t, t].
//
// A step is three launches: k_key_logits (the reuse decision and, when the step
// retrieves, one read of K; score.cu), k_vote_topk (score.cu; returns at once
// when the step reuses) and k_dec_attn. Whether the step retrieves is decided
// on the device, so a step never synchronises with the host.
#include <cuda_bf16.h>

#include <cmath>

#include "launch.cuh"
#include "ptx_sm103.cuh"
#include "scale_internal.h"
#include "score.cuh"

namespace scale {
namespace {

using namespace scale_ptx;

// Decode cache layout (bytes from its base).
constexpr size_t kDecState = 0;     // int32[8]: valid, steps, retrieve, -, anchor position
constexpr size_t kDecUnits = 64;    // int32[2] unit table [t, t + 1] of the anchor, int32 n_units
constexpr size_t kDecAnchor = 256;  // fp32 [H_q * 128]
// selection int32 [k] and its count follow the anchor

// Read-only 16-byte load; volatile keeps a run of them issued back to back.
__device__ __forceinline__ uint4 ld_nc(const uint4* p)
{
    uint4 r;
    asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
                 : "l"(p));
    return r;
}

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

constexpr int kDecMaxSplits = 64;  // key splits of a KV head
// Threads of an attention CTA: one CTA of 512 per SM where a thread's 128
// registers hold its G query heads, else 256. Half as many CTAs of twice the
// size leave half the partials for the CTA that merges them.
template <int G>
constexpr int dec_threads = G <= 4 ? 512 : 256;

struct DecArgs {
    int Hq, Hkv;
    int64_t t;          // position of the decode query (its K and V rows are present)
    int n_sink, n_local, k;
    float attn_scale_log2;
    int32_t* state;     // valid, steps sharing the anchor, retrieved, -, anchor position
    int32_t* units;     // [t_anchor, t_anchor + 1], then 1
    float* anchor;
    const int32_t* sel;
    const int32_t* sel_count;
    const int32_t* gate;  // 1 when the step retrieves
    int32_t* tickets;     // [H_kv], zero at the start of the step
    float4* o_part;       // [H_q][kDecMaxSplits][32] unnormalised outputs
    float2* ml_part;      // [H_q][kDecMaxSplits] (max, sum)
    int splits;
};

__host__ __device__ __forceinline__ int64_t window_start(int n_local, int64_t t)
{
    return t - n_local > 0 ? t - n_local : 0;
}

// Attention of the query over its keys: key i of the step is the sink i
// (i < n_s = min(n_sink, W_t)), then the cached selection (produced by the
// top-k: ascending, inside [n_sink, W_a) with W_a <= W_t), then the window
// [W_t, t]. Grid (KV heads, key splits). A half-warp takes a key for all G
// query heads of the KV head: lane c holds dimensions [8 c, 8 c + 8), so a K
// or V row is one 256-byte read of the half-warp, read once for the G heads,
// and the rows of KB keys are in flight per online-softmax update (log2
// units). The 16 partial dot products of an update are added over the lanes by
// halving exchanges (15 shuffles instead of 64), which leaves each (head, key)
// pair in one lane: it takes one exponential. The CTA's half-warps are merged in
// order in shared memory; the CTA that finishes last for a KV head (a ticket
// counter) merges the splits of its heads in order and writes the bf16 output.
// Bound by latency and issue: 38 MB of K and V at k = 8192 (5.6 us of HBM time)
// take 17 us alone with cold caches (before: a warp per head and a combine kernel, 44 us).
// Also stores what the step's reuse decision changes: the state words and, when
// the step retrieved, the anchor.
template <int G>
__global__ void __launch_bounds__(dec_threads<G>, 1) k_dec_attn(const DecArgs a, const __nv_bfloat16* __restrict__ q,
                                                          const uint4* __restrict__ k,
                                                          const uint4* __restrict__ v,
                                                          __nv_bfloat16* __restrict__ out)
{
    constexpr int kDecThreads = dec_threads<G>;
    constexpr int kDecWarps = kDecThreads / 32;
    constexpr int kDecStep = 2 * kDecWarps;  // half-warps of the CTA
    constexpr int KB = G <= 2 ? 8 : G <= 4 ? 4 : 2;  // keys per half-warp and update: G KB <= 16
    __shared__ float s_o[kDecWarps][G][kHeadDim];
    __shared__ float2 s_ml[kDecWarps][G];
    __shared__ float s_w[G][kDecMaxSplits];
    __shared__ int s_last;
    pdl_enter();
    const int j = blockIdx.x, split = blockIdx.y;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int half = lane >> 4, c = lane & 15;
    const bool retrieved = *a.gate != 0;
    if (j == 0 && split == 0 && tid == 0) {
        if (retrieved) {
            a.state[0] = 1;
            a.state[1] = 1;
            a.state[4] = static_cast<int32_t>(a.t);
            a.units[0] = static_cast<int32_t>(a.t);
            a.units[1] = static_cast<int32_t>(a.t + 1);
            a.units[2] = 1;
        } else {
            a.state[1] += 1;
        }
        a.state[2] = retrieved;
    }
    if (retrieved && split == 0)
        for (int i = tid; i < G * kHeadDim; i += kDecThreads)
            a.anchor[j * G * kHeadDim + i] = __bfloat162float(q[j * G * kHeadDim + i]);

    const int64_t W = window_start(a.n_local, a.t);
    const int n_s = static_cast<int>(a.n_sink < W ? a.n_sink : W);
    int n_sel = *a.sel_count;
    n_sel = n_sel < 0 ? 0 : (n_sel > a.k ? a.k : n_sel);
    const int n = n_s + n_sel + static_cast<int>(a.t - W + 1);
    const int i0 = static_cast<int>(static_cast<int64_t>(n) * split / a.splits);
    const int i1 = static_cast<int>(static_cast<int64_t>(n) * (split + 1) / a.splits);
    auto token_of = [&](int i) -> int64_t {
        return i < n_s ? i : (i < n_s + n_sel ? a.sel[i - n_s] : W + (i - n_s - n_sel));
    };
    uint32_t qw[G][4];  // bf16 pairs
#pragma unroll
    for (int hl = 0; hl < G; ++hl) {
        const uint4 x = *reinterpret_cast<const uint4*>(q + (j * G + hl) * kHeadDim + 8 * c);
        qw[hl][0] = x.x;
        qw[hl][1] = x.y;
        qw[hl][2] = x.z;
        qw[hl][3] = x.w;
    }
    float o[G][8];
#pragma unroll
    for (int hl = 0; hl < G; ++hl)
#pragma unroll
        for (int e = 0; e < 8; ++e) o[hl][e] = 0.f;
    // Lane c of a half-warp also keeps the softmax of key c % KB of every KB
    // for head c / KB: the running max of the head, its own keys' sum.
    float m = -INFINITY, l = 0.f;
    const int u_l = c % KB;
    const uint4 zero = make_uint4(0, 0, 0, 0);
    // half-warp x of the CTA takes the keys i0 + x, i0 + x + kDecStep, ...; lane c
    // looks up the token of the half-warp's key c of every 16
    for (int b0 = i0 + 2 * warp; b0 < i1; b0 += 16 * kDecStep) {  // warp-uniform
        const int ic = b0 + half + kDecStep * c;
        const int64_t tok = ic < i1 ? token_of(ic) : -1;
        for (int r0 = 0; r0 < 16 && b0 + kDecStep * r0 < i1; r0 += KB) {  // warp-uniform
            uint4 kw[KB], vw[KB];
#pragma unroll
            for (int u = 0; u < KB; ++u) {
                const int64_t t = __shfl_sync(0xFFFFFFFFu, tok, half * 16 + r0 + u);
                const int64_t row = (t * a.Hkv + j) * 16 + c;
                kw[u] = t < 0 ? zero : ld_nc(k + row);
                vw[u] = t < 0 ? zero : ld_nc(v + row);
            }
            // this lane's 8 dimensions of q . k for (head, key) pair hl * KB + u ...
            float s[16];
#pragma unroll
            for (int x = 0; x < 16; ++x) s[x] = 0.f;
#pragma unroll
            for (int u = 0; u < KB; ++u) {
                const uint32_t w[4] = {kw[u].x, kw[u].y, kw[u].z, kw[u].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float klo = bf16_lo(w[e]), khi = bf16_hi(w[e]);
#pragma unroll
                    for (int hl = 0; hl < G; ++hl)
                        s[hl * KB + u] = fmaf(bf16_lo(qw[hl][e]), klo, fmaf(bf16_hi(qw[hl][e]), khi, s[hl * KB + u]));
                }
            }
            // ... added over the 16 lanes so that lane c ends with pair c's sum
#pragma unroll
            for (int x = 8; x > 0; x >>= 1)
#pragma unroll
                for (int y = 0; y < x; ++y) {
                    const float keep = (c & x) ? s[y + x] : s[y];
                    const float give = (c & x) ? s[y] : s[y + x];
                    s[y] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, x);
                }
            const float sl = b0 + half + kDecStep * (r0 + u_l) < i1 ? s[0] * a.attn_scale_log2 : -INFINITY;
            float m_new = sl;
#pragma unroll
            for (int x = 1; x < KB; x <<= 1) m_new = fmaxf(m_new, __shfl_xor_sync(0xFFFFFFFFu, m_new, x));
            m_new = fmaxf(m, m_new);
            const float base = m_new == -INFINITY ? 0.f : m_new;
            const float alpha = ex2(m - base);
            const float p = ex2(sl - base);
            l = l * alpha + p;
            if (__any_sync(0xFFFFFFFFu, m != m_new)) {
#pragma unroll
                for (int hl = 0; hl < G; ++hl) {
                    const float f = __shfl_sync(0xFFFFFFFFu, alpha, half * 16 + hl * KB);
#pragma unroll
                    for (int e = 0; e < 8; ++e) o[hl][e] *= f;
                }
            }
            m = m_new;
#pragma unroll
            for (int u = 0; u < KB; ++u) {
                const uint32_t w[4] = {vw[u].x, vw[u].y, vw[u].z, vw[u].w};
#pragma unroll
                for (int hl = 0; hl < G; ++hl) {
                    const float pu = __shfl_sync(0xFFFFFFFFu, p, half * 16 + hl * KB + u);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        o[hl][2 * e] = fmaf(pu, bf16_lo(w[e]), o[hl][2 * e]);
                        o[hl][2 * e + 1] = fmaf(pu, bf16_hi(w[e]), o[hl][2 * e + 1]);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int x = 1; x < KB; x <<= 1) l += __shfl_xor_sync(0xFFFFFFFFu, l, x);  // the head's sum
    // the warp's two halves, then the warps in order
#pragma unroll
    for (int hl = 0; hl < G; ++hl) {
        const float m1 = __shfl_sync(0xFFFFFFFFu, m, half * 16 + hl * KB);
        const float m2 = __shfl_sync(0xFFFFFFFFu, m, (half ^ 1) * 16 + hl * KB);
        const float l1 = __shfl_sync(0xFFFFFFFFu, l, half * 16 + hl * KB);
        const float l2 = __shfl_sync(0xFFFFFFFFu, l, (half ^ 1) * 16 + hl * KB);
        const float mm = fmaxf(m1, m2);
        const float base = mm == -INFINITY ? 0.f : mm;
        const float w1 = ex2(m1 - base), w2 = ex2(m2 - base);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float o2 = __shfl_xor_sync(0xFFFFFFFFu, o[hl][e], 16);
            if (half == 0) s_o[warp][hl][8 * c + e] = o[hl][e] * w1 + o2 * w2;
        }
        if (lane == 0) s_ml[warp][hl] = make_float2(mm, l1 * w1 + l2 * w2);
    }
    __syncthreads();
    for (int x = tid; x < G * kHeadDim; x += kDecThreads) {
        const int hl = x / kHeadDim, dd = x % kHeadDim;
        float mm = -INFINITY;
#pragma unroll
        for (int w = 0; w < kDecWarps; ++w) mm = fmaxf(mm, s_ml[w][hl].x);
        const float base = mm == -INFINITY ? 0.f : mm;
        float ll = 0.f, oo = 0.f;
#pragma unroll
        for (int w = 0; w < kDecWarps; ++w) {
            const float f = ex2(s_ml[w][hl].x - base);
            ll += s_ml[w][hl].y * f;
            oo += s_o[w][hl][dd] * f;
        }
        const int64_t slot = static_cast<int64_t>(j * G + hl) * kDecMaxSplits + split;
        __stcg(reinterpret_cast<float*>(a.o_part + slot * 32) + dd, oo);
        if (dd == 0) __stcg(&a.ml_part[slot], make_float2(mm, ll));
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&a.tickets[j], 1) == a.splits - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // every split of KV head j is stored: weights 2^(m_s - m) / l, then the sum
    for (int hl = warp; hl < G; hl += kDecWarps) {
        const float2* ml = a.ml_part + static_cast<int64_t>(j * G + hl) * kDecMaxSplits;
        float2 x[kDecMaxSplits / 32];
        float mm = -INFINITY, ll = 0.f;
#pragma unroll
        for (int e = 0; e < kDecMaxSplits / 32; ++e) {
            const int sp = lane + 32 * e;
            x[e] = sp < a.splits ? __ldcg(&ml[sp]) : make_float2(-INFINITY, 0.f);
            mm = fmaxf(mm, x[e].x);
        }
        for (int y = 16; y > 0; y >>= 1) mm = fmaxf(mm, __shfl_xor_sync(0xFFFFFFFFu, mm, y));
        const float base = mm == -INFINITY ? 0.f : mm;
#pragma unroll
        for (int e = 0; e < kDecMaxSplits / 32; ++e) ll += x[e].y * ex2(x[e].x - base);
        for (int y = 16; y > 0; y >>= 1) ll += __shfl_xor_sync(0xFFFFFFFFu, ll, y);
        const float inv = ll > 0.f ? 1.0f / ll : 0.f;
#pragma unroll
        for (int e = 0; e < kDecMaxSplits / 32; ++e) s_w[hl][lane + 32 * e] = ex2(x[e].x - base) * inv;
    }
    __syncthreads();
    // warp w sums the splits w, w + kDecWarps, ... of every head; s_o takes the warps' sums
    float4 acc[G];
#pragma unroll
    for (int hl = 0; hl < G; ++hl) acc[hl] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
    for (int sp = warp; sp < a.splits; sp += kDecWarps)
#pragma unroll
        for (int hl = 0; hl < G; ++hl) {
            const float4 x = __ldcg(&a.o_part[(static_cast<int64_t>(j * G + hl) * kDecMaxSplits + sp) * 32 + lane]);
            const float w = s_w[hl][sp];
            acc[hl].x += x.x * w;
            acc[hl].y += x.y * w;
            acc[hl].z += x.z * w;
            acc[hl].w += x.w * w;
        }
#pragma unroll
    for (int hl = 0; hl < G; ++hl) *reinterpret_cast<float4*>(&s_o[warp][hl][4 * lane]) = acc[hl];
    __syncthreads();
    for (int x = tid; x < G * kHeadDim; x += kDecThreads) {
        const int hl = x / kHeadDim, d = x % kHeadDim;
        float r = 0.f;
#pragma unroll
        for (int w = 0; w < kDecWarps; ++w) r += s_o[w][hl][d];
        out[(j * G + hl) * kHeadDim + d] = __float2bfloat16_rn(r);
    }
}

template <int G>
cudaError_t run_dec_attn(const DecArgs& a, const void* q, const void* k, const void* v, void* out, cudaStream_t st)
{
    return launch_after(st, dim3(a.Hkv, a.splits), dec_threads<G>, 0, 1, k_dec_attn<G>, a,
                        static_cast<const __nv_bfloat16*>(q), static_cast<const uint4*>(k),
                        static_cast<const uint4*>(v), static_cast<__nv_bfloat16*>(out));
}

// Keys per (max, sum) pair of the logits that the workspace has room for.
constexpr int kDecStat = 64;

// Regions of the decode workspace (byte offsets from its base; the status word
// comes first).
struct DecWs {
    size_t z;        // fp32 [H_q][z_stride]               logits, rows padded to four tokens
    size_t zpart;    // float2 [H_q][n_stat]               partial softmax sums of the logits
    size_t o_part;   // float4 [H_q][kDecMaxSplits][32]    attention: unnormalised outputs
    size_t ml_part;  // float2 [H_q][kDecMaxSplits]        (max, sum)
    size_t tickets;  // int32 [H_kv], then the gate
    size_t scratch;  // int32 [kVoteScratchInts]           vote and top-k
    size_t end;
    int64_t z_stride, n_stat;
};

DecWs decode_layout(const Derived& d)
{
    DecWs w{};
    size_t off = 256;
    auto take = [&](size_t bytes) {
        const size_t at = off;
        off = align_up(off + bytes, kAlign);
        return at;
    };
    const size_t heads = static_cast<size_t>(d.Hq);
    w.z_stride = (d.N + 3) / 4 * 4;
    w.n_stat = (d.N + kDecStat - 1) / kDecStat;
    w.z = take(heads * w.z_stride * sizeof(float));
    w.zpart = take(heads * w.n_stat * sizeof(float2));
    w.o_part = take(heads * kDecMaxSplits * kHeadDim * sizeof(float));
    w.ml_part = take(heads * kDecMaxSplits * sizeof(float2));
    w.tickets = take((static_cast<size_t>(d.Hkv) + 1) * sizeof(int32_t));
    w.scratch = take(kVoteScratchInts * sizeof(int32_t));
    w.end = off;
    return w;
}

}  // namespace

size_t decode_cache_bytes(const Derived& d)
{
    return kDecAnchor + static_cast<size_t>(d.Hq) * kHeadDim * sizeof(float) +
           static_cast<size_t>(d.k > 0 ? d.k : 1) * sizeof(int32_t) + 256;
}

// The size that callers are told, and may have stored: more than the regions
// take (65 KB a head beside the logits and their sums, of which they take less
// than half, and 27 KB once).
size_t decode_ws_bytes(const Derived& d)
{
    constexpr size_t kHeadBytes = 128 * 130 * sizeof(float);
    const size_t cap = static_cast<size_t>(d.N), heads = static_cast<size_t>(d.Hq);
    size_t off = 256;
    for (const size_t bytes : {heads * cap * sizeof(float), heads * sizeof(float2), cap * sizeof(float), heads * kHeadBytes,
                               heads * ((cap + kDecStat - 1) / kDecStat) * sizeof(float2),
                               (kTopkPasses * 256 + (kTopkPasses + 1) * 4) * sizeof(int32_t),
                               static_cast<size_t>(topk_max_chunks(d)) * sizeof(int2)})
        off = align_up(off + bytes, kAlign);
    const size_t end = decode_layout(d).end;
    return off > end ? off : end;
}

cudaError_t launch_decode_step(const Derived& d, int64_t t, const void* q, const void* k, const void* v,
                               uint8_t* cache, void* out, uint8_t* ws, uint64_t timeout_ns, cudaStream_t st)
{
    auto* state = reinterpret_cast<int32_t*>(cache + kDecState);
    auto* anchor = reinterpret_cast<float*>(cache + kDecAnchor);
    auto* sel = reinterpret_cast<int32_t*>(cache + kDecAnchor + static_cast<size_t>(d.Hq) * kHeadDim * sizeof(float));
    int32_t* sel_count = sel + (d.k > 0 ? d.k : 1);
    auto* status = reinterpret_cast<int32_t*>(ws + kStatusOffset);
    const DecWs lay = decode_layout(d);
    auto* z = reinterpret_cast<float*>(ws + lay.z);
    auto* zpart = reinterpret_cast<float2*>(ws + lay.zpart);
    auto* gate = reinterpret_cast<int32_t*>(ws + lay.tickets) + d.Hkv;
    auto* scratch = reinterpret_cast<int32_t*>(ws + lay.scratch);

    DecArgs a;
    a.Hq = d.Hq;
    a.Hkv = d.Hkv;
    a.t = t;
    a.n_sink = d.n_sink;
    a.n_local = d.n_local;
    a.k = d.k;
    a.attn_scale_log2 = d.attn_scale * 1.4426950408889634f;
    a.state = state;
    a.units = reinterpret_cast<int32_t*>(cache + kDecUnits);
    a.anchor = anchor;
    a.sel = sel;
    a.sel_count = sel_count;
    a.o_part = reinterpret_cast<float4*>(ws + lay.o_part);
    a.ml_part = reinterpret_cast<float2*>(ws + lay.ml_part);
    a.tickets = reinterpret_cast<int32_t*>(ws + lay.tickets);
    a.gate = gate;

    // One unit of one token, its position t (per-sub-chunk units with L = 1).
    const Units ut{nullptr, nullptr, 1, d.N, 1, static_cast<int>(d.N)};
    KeyScoreArgs s{};
    s.ut = ut;
    s.sc_begin = static_cast<int>(t);
    s.sc_end = static_cast<int>(t + 1);
    s.Hq = d.Hq;
    s.Hkv = d.Hkv;
    s.N = static_cast<int>(d.N);
    s.n_sink = d.n_sink;
    s.n_local = d.n_local;
    s.scale2 = d.sigma * 1.4426950408889634f;
    s.z = z;
    s.z_stride = lay.z_stride;
    s.part = zpart;
    s.scratch = scratch;
    s.status = status;
    s.timeout_ns = timeout_ns;
    s.pg = KvPaging{nullptr, 0, 0, d.N, d.N};
    s.q = q;
    s.anchor = anchor;
    s.state = state;
    s.S_max = d.S_max;
    s.theta = d.theta;
    s.gate = gate;
    s.tickets = a.tickets;
    const int64_t W = window_start(d.n_local, t);
    const bool any = W > d.n_sink;
    s.n_part = any ? key_logits_parts(W - d.n_sink / 128 * 128, d.Hkv, lay.n_stat) : 1;
    cudaError_t e = launch_key_logits(s, d.g, true, q, 1, k, 1, st);
    if (e != cudaSuccess) return e;
    if (any) {
        VoteArgs w{};
        w.ut = ut;
        w.sc_begin = s.sc_begin;
        w.sc_end = s.sc_end;
        w.Hq = d.Hq;
        w.g = d.g;
        w.N = s.N;
        w.k = d.k;
        w.n_sink = d.n_sink;
        w.n_local = d.n_local;
        w.scale2 = s.scale2;
        w.z = z;
        w.z_stride = lay.z_stride;
        w.part = zpart;
        w.n_part = s.n_part;
        w.scores = nullptr;
        w.sel = sel;
        w.sel_count = sel_count;
        w.single = 1;
        w.scratch = scratch;
        w.gate = gate;
        w.status = status;
        w.timeout_ns = timeout_ns;
        e = launch_vote_topk(w, st);
    } else {
        // no candidates: the selection is empty whenever this step retrieves
        e = cudaMemsetAsync(sel_count, 0, sizeof(int32_t), st);
    }
    if (e != cudaSuccess) return e;

    // Splits: at most one CTA per SM (one and two KV heads: kDecMaxSplits each), and
    // at least 64 keys each.
    int sms = 0;
    if ((e = device_sms(&sms)) != cudaSuccess) return e;
    const int64_t n_max = d.n_sink + static_cast<int64_t>(d.k) + (t - W + 1);
    int64_t splits = sms / d.Hkv;
    if (splits > (n_max + 63) / 64) splits = (n_max + 63) / 64;
    if (splits > kDecMaxSplits) splits = kDecMaxSplits;
    a.splits = static_cast<int>(splits > 0 ? splits : 1);
    switch (d.g) {
    case 1: return run_dec_attn<1>(a, q, k, v, out, st);
    case 2: return run_dec_attn<2>(a, q, k, v, out, st);
    case 3: return run_dec_attn<3>(a, q, k, v, out, st);
    case 4: return run_dec_attn<4>(a, q, k, v, out, st);
    case 5: return run_dec_attn<5>(a, q, k, v, out, st);
    case 6: return run_dec_attn<6>(a, q, k, v, out, st);
    case 7: return run_dec_attn<7>(a, q, k, v, out, st);
    case 8: return run_dec_attn<8>(a, q, k, v, out, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace scale
