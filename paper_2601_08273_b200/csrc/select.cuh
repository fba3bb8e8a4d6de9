// Arguments shared by the selection kernels (select.cu: fp64 scores of fp32 embeddings, fusion, top-k; select_gram.cu: scores of
// bf16 embeddings on the integer tensor path).
#pragma once

#include "common.cuh"

namespace hippo {

constexpr int kMaxCrop = 32;       // tokens per crop
constexpr int kSelMaxBatch = 64;   // sequences per call (kernel-parameter tables)

struct SelectParams {
    const void *embeds;
    const float *attn_mass;
    float *fused;
    int32_t *kept;
    double *norm2, *tdot, *s_spa;   // [total tokens]: squared norm, product with the next frame's, Eq. 5-6
    int cosines;                    // 1: tdot holds the cosine itself (the integer path), norm2 nothing
    int batch, grid_h, grid_w, crop_h, crop_w, d, tpf, crops_y, crops_x;
    unsigned mask;
    int seq_off[kSelMaxBatch + 1];    // token offset of each sequence
    int frame_off[kSelMaxBatch + 1];  // frame offset of each sequence
    int k[kSelMaxBatch];
    int k_off[kSelMaxBatch + 1];
    int *frame_budget;               // per-frame policy: [frames] tokens kept / [frames] first output position
    int *frame_out;
};

__device__ __forceinline__ int find_seq(const int *off, int n, int x) {  // largest b with off[b] <= x
    int b = 0;
    while (b + 1 < n && off[b + 1] <= x) ++b;
    return b;
}

// C[8 x 8] += A[8 x 4] B[4 x 8]: lane holds A[lane / 4][lane % 4], B[lane % 4][lane / 4], C[lane / 4][lane % 4 * 2 + {0, 1}]
__device__ __forceinline__ void dmma_m8n8k4(double &c0, double &c1, double a, double b) {
    asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
                 : "+d"(c0), "+d"(c1) : "d"(a), "d"(b));
}

// norms, temporal dot products and spatial scores of bf16 embeddings (norm2, tdot, s_spa of p)
constexpr int kGramMaxDim = 65536;   // 32-bit sums of digit products, 16-bit positions in the list of large elements
int32_t select_gram_cost(const SelectParams &p, double &us);   // about how long its tiles take
int32_t launch_select_gram(const SelectParams &p, WsHeader *header, cudaStream_t stream);

}  // namespace hippo
