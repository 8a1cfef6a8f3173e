// Decode-time attention over the cache (Section 3.4): declarations.
#pragma once
#include "common.cuh"

namespace freqkv {

constexpr int ATTEND_MAX_BATCH = 128;  // sequences per launch (lengths travel as kernel arguments)

bool attend_supported(int32_t head_dim, int32_t q_heads_per_kv);
// How the rows of every (sequence, kv head) are split.
struct AttendPlan {
    int32_t chunk;    // most rows of one CTA
    int32_t splits;   // of the longest sequence
    bool one_wave;    // all CTAs are resident at once
    bool captured;    // the launches go into a graph: no tickets, no overlap with the launch before
};
AttendPlan attend_plan(int32_t batch, const int32_t* lens, int32_t kv_heads, int32_t q_heads_per_kv, int32_t dtype, int sm_count);
// No plan for lengths up to `longest` has more splits (unless rows beyond what 64 CTAs can take force them).
int32_t attend_most_splits(int32_t longest);
// Work areas: one ticket per (sequence, kv head) of a call whose CTAs are all resident, zero before the first launch and
// after every launch; the splits' partials.
size_t attend_ticket_bytes(int sm_count);
size_t attend_partial_bytes(int32_t splits, int32_t batch, int32_t q_heads);
// table[pos][c] = (cos, sin)(pos * base^(-2c/128)), pos < rows, c < 64.
cudaError_t launch_rope_table(float2* table, int32_t rows, double base, cudaStream_t stream);
// q, out: [batch, kv_heads * g, 128] in the cache dtype; table may be null (no RoPE).
cudaError_t launch_attend(const freqkv_layout& l, const void* k, const void* v, int32_t layer, const void* q, void* out,
                          int32_t g, const int32_t* lens_host, const float2* table, float scale, const AttendPlan& plan,
                          float* partial, int32_t* tickets, int32_t* launched, cudaStream_t stream);

}  // namespace freqkv
