// score.cuh -- arguments and launchers of the few-unit selection at block size
// 1 (score.cu), used by the token-level selection and by the decode step.
#pragma once

#include <cuda_bf16.h>

#include "scale_internal.h"

namespace scale {

constexpr int kVoteBins = 2048;        // radix digits of 11, 11 and 10 bits
constexpr int kVoteGroup = 8;          // planes loaded together by the vote
constexpr int kVoteMaxCtas = 256;
// Scratch of one unit (int32 words): the three passes' histograms, the barrier
// counter, and the CTAs' (above, equal) counts. k_key_logits clears all but the
// counts.
constexpr int kVoteCounter = 3 * kVoteBins;
constexpr int kVoteCounts = kVoteCounter + 16;
constexpr int kVoteScratchInts = kVoteCounts + 2 * kVoteMaxCtas;

struct KeyScoreArgs {
    Units ut;
    int sc_begin, sc_end;
    int Hq, Hkv;
    int N;
    int64_t z_stride;   // floats between the heads' planes, a multiple of 4
    int n_sink, n_local;
    float scale2;       // sigma * log2(e)
    float* z;           // [units][H_q][z_stride]
    float2* part;       // [units][H_q][n_part] (m, sum of 2^(z scale2 - m))
    int n_part;
    int32_t* scratch;   // [units][kVoteScratchInts]
    int32_t* status;
    uint64_t timeout_ns;
    KvPaging pg;
    // decode step only
    const void* q;         // bf16 [H_q][128]
    const float* anchor;   // fp32 [H_q][128]
    const int32_t* state;  // valid, steps sharing the anchor
    int S_max;
    float theta;
    int32_t* gate;         // out: 1 when the step retrieves
    int32_t* tickets;      // [H_kv] cleared for the attention kernel
};

struct VoteArgs {
    Units ut;
    int sc_begin, sc_end;
    int Hq, g, N, k, n_sink, n_local;
    float scale2;
    float* z;
    int64_t z_stride;
    const float2* part;
    int n_part;
    float* scores;         // [M][N] or null
    int32_t* sel;          // row u (row 0 when `single`)
    int32_t* sel_count;
    int single;
    int32_t* scratch;
    const int32_t* gate;   // null, or run only when *gate != 0
    int32_t* status;
    uint64_t timeout_ns;
};

// CTAs per unit tile of k_key_logits (= partials per head): two per SM, at most
// one per (128-key tile, KV head) and at most `room`.
int key_logits_parts(int64_t cand_end, int Hkv, int64_t room);
// `operand`: bf16 [3][H_kv][M][g][128] fingerprint parts, or the bf16 query
// [H_q][128] of a decode step.
cudaError_t launch_key_logits(const KeyScoreArgs& a, int g, bool decode, const void* operand, int64_t M,
                              const void* k, int max_units, cudaStream_t st);
cudaError_t launch_vote_topk(const VoteArgs& a, cudaStream_t st);

}  // namespace scale
