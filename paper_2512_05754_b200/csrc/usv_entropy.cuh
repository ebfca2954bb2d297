// Arguments of the key-marginal kernel (Sec. 3.4, Eq. 16) and its launcher.
#pragma once
#include "usv_common.cuh"

namespace usv {

struct MargArgs {
    const __nv_bfloat16 *q, *k;
    usv_strides sq, sk;
    const int32_t* sel;
    const float* lse;     // [B,H,N] natural log of the softmax denominator (incl. the max)
    float* marg;          // [B,N], zeroed before the launch
    unsigned int* status; // device status word the bounded waits report to (may be NULL)
    int B, H, N, NB, kmax;
    float scale_log2;     // softmax scale * log2(e)
    float inv_hn;         // 1 / (H N)
    int k_per_head[USV_MAX_HEADS];
    // Pairs of query blocks and their union lists as usv_attn_plan.cu writes them; NULL: neighbours are paired.
    const int2* pairs;
    const int* lists;
    int64_t list_batch, list_off[USV_MAX_HEADS];
};

// usv_entropy_tc.cu; marg must be zero.
int launch_marginal_tc(const MargArgs& a, int d, cudaStream_t st);
// whether a pairing plan pays for the call
bool marginal_planned(const MargArgs& a, int sms);
// room for the plan of any call with lists of at most kmax blocks; 0 where none of them pays
size_t marginal_plan_bytes(int B, int H, int NB, int kmax);
size_t pair_plan_bytes(int B, int H, int NB, const int32_t* k_per_head);
// Enqueues the plan of the call in mem and points a to it.
int launch_marginal_plan(MargArgs& a, void* mem, cudaStream_t st);

}  // namespace usv
