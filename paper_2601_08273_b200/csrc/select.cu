// hippo_select_tokens: semantic-aware visual-token preservation (Section 5.1).
//
//   Eq. 3-4  s_temp(j) = 1 - mean over the adjacent frames that contain j's grid cell of cos(v_j^f, v_j^f')
//   Eq. 5-6  s_spa(j)  = (1/M) sum_k (S_jk - mu_j)^2 over the M tokens of j's crop, S = cosine Gram matrix, S_jj = 1
//   Eq. 7    fused = z(attn) + z(spa) + z(temp), z = per-frame standardisation with the population sigma
//   top-k    k best over the sequence by (fused as fp32 descending, index ascending), emitted ascending
//
// The standardisation of s_spa divides by a sigma of ~1e-4 on near-orthogonal embeddings, which magnifies any
// rounding in the Gram entries by four orders of magnitude.  All dot products, crop statistics and frame
// statistics therefore have the accuracy of fp64 sums (bf16 x bf16 products are exact in fp64), so the kept set only
// depends on the final rounding of the fused score to fp32.
//
// Kernels:  bf16: gram (select_gram.cu: norms, next-frame dots and spatial scores from integer tensor instructions);
//           fp32, small bf16 calls and calls without the spatial term: dots (norms + next-frame dot, one warp per token) -> spatial (one CTA per crop, fp64
//           tensor instructions);  then fuse (one CTA per frame: s_temp, three standardisations, sum) -> topk (one cluster of
//           CTAs per sequence, histograms of the digits of order-preserving keys, ordered compaction).
//
// hippo_select_tokens_policy adds the selection rules the paper compares itself with, as rules only: a uniform budget
// per frame (the attention-guided uniform pruning of earlier video speculative decoding, related-work section), the k
// best by caller-supplied random keys and whole frames at a regular stride (exploration of pruning criteria,
// Section 6).  Uniform: budgets by one thread per sequence, then one CTA per frame ranks its tokens by counting.
#include <math.h>

#include <type_traits>

#include "select.cuh"
#include "tc_ptx.cuh"

namespace hippo {

__device__ __forceinline__ double ld_as_double(const float *p, size_t i) { return (double)p[i]; }
__device__ __forceinline__ double ld_as_double(const __nv_bfloat16 *p, size_t i) { return (double)__bfloat162float(p[i]); }

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ---- norms and the dot product with the same cell of the next frame ------------------------------------------
template <typename T> __device__ __forceinline__ void load8(const T *p, double *v);
template <> __device__ __forceinline__ void load8<__nv_bfloat16>(const __nv_bfloat16 *p, double *v) {
    const uint4 u = __ldg(reinterpret_cast<const uint4 *>(p));
    const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&u);
#pragma unroll
    for (int i = 0; i < 4; ++i) { const float2 f = __bfloat1622float2(h[i]); v[2 * i] = (double)f.x; v[2 * i + 1] = (double)f.y; }
}
template <> __device__ __forceinline__ void load8<float>(const float *p, double *v) {
    const float4 a = __ldg(reinterpret_cast<const float4 *>(p)), c = __ldg(reinterpret_cast<const float4 *>(p) + 1);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = c.x; v[5] = c.y; v[6] = c.z; v[7] = c.w;
}

// One warp per token; a lane takes 8 consecutive elements per step (embed_dim is a multiple of 8).
constexpr int kDotsThreads = 256;
template <typename T>
__device__ __forceinline__ void select_dots(const SelectParams &p, int block) {
    const int total = p.seq_off[p.batch];
    const int j = block * (kDotsThreads / 32) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (j >= total) return;
    const int b = find_seq(p.seq_off, p.batch, j);
    const T *E = (const T *)p.embeds;
    const size_t a = (size_t)j * p.d;
    const bool has_next = j + p.tpf < p.seq_off[b + 1];
    const size_t c = a + (size_t)p.tpf * p.d;
    double n2 = 0.0, td = 0.0;
    for (int i = lane * 8; i < p.d; i += 256) {
        double x[8], y[8];
        load8(E + a + i, x);
        if (has_next) load8(E + c + i, y);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            n2 = fma(x[e], x[e], n2);
            if (has_next) td = fma(x[e], y[e], td);
        }
    }
    n2 = warp_sum(n2);
    td = warp_sum(td);
    if (lane == 0) { p.norm2[j] = n2; p.tdot[j] = td; }
}
template <typename T>
__global__ void __launch_bounds__(kDotsThreads) select_dots_kernel(const SelectParams p) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    select_dots<T>(p, (int)blockIdx.x);
}

// ---- spatial score on the fp64 tensor path: one CTA per crop ---------------------------------------------------------
// The Gram matrix of the crop's embeddings is a dense fp64 contraction over the embedding dimension: it runs on
// mma.sync.m8n8k4.f64 (exact fp64 products of the widened inputs, fp64 accumulation; measured on B200: one instruction per
// 16.1 clocks and SM quarter, i.e. 63.6 multiply-adds per clock and SM, whatever the operand values and also with the
// operands read from shared memory and widened on the way).  Tokens are taken in groups of eight; for the groups a <= c the
// 8 x 8 tile G[a][c] needs one fragment per group and step of four dimensions, and for a Gram matrix the A fragment of a
// group (row = lane / 4, dimension = lane % 4) is also its B fragment.  Warp w owns dimensions [16 w, 16 w + 16) of every
// 128-dimension chunk: it stages them itself, in the storage type, straight from global memory with cp.async into a ring
// of its own (rows back to back, so the eight rows of a fragment load are contiguous), and waits for nobody else's
// copies: there is no block-wide barrier inside the loop.  Since the order of a dot product's terms is free, lane l takes
// dimensions 4 (l % 4) .. + 3 of the warp's sixteen: one 8-byte (bf16) load per group and chunk, widened to fp64 in
// registers, feeds the four steps.  Every staged element is read exactly once.  The eight warps' tiles are added in shared
// memory at the end, in a fixed order; the diagonal of G holds the squared norms.
// The multiply sequence is instantiated per number of groups: with the group count a run-time value every instruction of
// it sat behind a branch of its own and the pipe was busy half of the time (32k tokens, whole selection: 472 us with the
// branches, 351 us without, 343 us with the warps' own rings).
// A crop of 8 n + 1 tokens (the paper's 5 x 5 = 25) would pay n + 1 tiles for its last token: that token's dot products
// come from plain multiply-adds on the fragments the lane holds anyway (see below).
constexpr int kMmaChunk = 128;                 // dimensions per chunk, over the eight warps
constexpr int kMmaWarpDims = 16;               // dimensions of a chunk that one warp stages and multiplies
constexpr int kMmaThreads = 256;
constexpr int kMmaWarps = kMmaThreads / 32;
constexpr int kMmaTiles = 10;                  // 4 groups: upper triangle incl. diagonal
static_assert(kMmaWarps * kMmaWarpDims == kMmaChunk, "the warps' slices make up a chunk");
template <typename T> struct MmaShape {
    static constexpr int kPiece = 16 / (int)sizeof(T);               // elements per 16-byte piece
    static constexpr int kPiecesPerRow = kMmaWarpDims / kPiece;
    static constexpr int kWarpRowBytes = kMmaWarpDims * (int)sizeof(T);   // rows back to back: the eight rows of a fragment load are contiguous
    static constexpr int kWarpStageBytes = kMaxCrop * kWarpRowBytes;
    static constexpr int kStages = 12 / (int)sizeof(T);              // 6 chunks in flight per warp (bf16), 3 (fp32): 6 KB per warp
    static constexpr size_t kWarpRingBytes = (size_t)kStages * kWarpStageBytes;
    static constexpr size_t kRingBytes = (size_t)kMmaWarps * kWarpRingBytes;
    static constexpr size_t kRedBytes = (size_t)kMmaWarps * kMmaTiles * 64 * sizeof(double);
    static constexpr size_t kSmemBytes = kRingBytes > kRedBytes ? kRingBytes : kRedBytes;
};

// 16 bytes global -> shared, asynchronously; n_bytes = 0 writes zeros and reads nothing
__device__ __forceinline__ void cp_async_16(void *dst, const void *src, int n_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(n_bytes) : "memory");
}
__device__ __forceinline__ void load_frag4(const __nv_bfloat16 *p, double *v) {
    const uint2 u = *reinterpret_cast<const uint2 *>(p);
    const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&u);
    const float2 a = __bfloat1622float2(h[0]), b = __bfloat1622float2(h[1]);
    v[0] = (double)a.x; v[1] = (double)a.y; v[2] = (double)b.x; v[3] = (double)b.y;
}
__device__ __forceinline__ void load_frag4(const float *p, double *v) {
    const float4 a = *reinterpret_cast<const float4 *>(p);
    v[0] = (double)a.x; v[1] = (double)a.y; v[2] = (double)a.z; v[3] = (double)a.w;
}

// The blocks behind the crops' form the norms and the products with the next frame, which need nothing of the crops: one launch for
// both (whole selection of 2,048 tokens of 1,024, bf16: 29.3 us with two, 27.4).
template <typename T>
__global__ void __launch_bounds__(kMmaThreads, 3) select_spatial_mma_kernel(const SelectParams p) {
    static_assert(kMmaThreads == kDotsThreads, "one launch for both");
    using Sh = MmaShape<T>;
    extern __shared__ __align__(16) uint8_t mma_smem[];   // ring of staged chunks; reused for the warps' partial tiles
    __shared__ int tok[kMaxCrop];
    __shared__ double S[kMaxCrop][kMaxCrop + 1];
    __shared__ double root[kMaxCrop];
    __shared__ double tail_red[kMmaWarps][kMaxCrop + 1];
    __shared__ int s_M;
    const int crops_per_frame = p.crops_y * p.crops_x, n_crops = p.frame_off[p.batch] * crops_per_frame;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if ((int)blockIdx.x >= n_crops) {
        select_dots<T>(p, (int)blockIdx.x - n_crops);
        return;
    }
    const int gframe = blockIdx.x / crops_per_frame, cr = blockIdx.x % crops_per_frame;
    const int b = find_seq(p.frame_off, p.batch, gframe);
    const int f = gframe - p.frame_off[b];
    const int n_v = p.seq_off[b + 1] - p.seq_off[b];
    const int nf = min(p.tpf, n_v - f * p.tpf);
    const int y0 = (cr / p.crops_x) * p.crop_h, x0 = (cr % p.crops_x) * p.crop_w;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        int M = 0;
        for (int y = y0; y < y0 + p.crop_h && y < p.grid_h; ++y)
            for (int x = x0; x < x0 + p.crop_w && x < p.grid_w; ++x)
                if (y * p.grid_w + x < nf) tok[M++] = p.seq_off[b] + f * p.tpf + y * p.grid_w + x;
        s_M = M;
    }
    __syncthreads();
    const int M = s_M;
    if (M == 0) return;
    const T *E = (const T *)p.embeds;
    if (M > 1) {
        // A crop of 8n + 1 tokens (the full 5 x 5 crop: 25) would pay a whole extra group, n + 1 tiles, for its last
        // token.  Its n * 8 dot products and its norm come from plain multiply-adds instead: at every step a lane already
        // holds, as tile operands, token (8g + lane / 4) at the step's dimension for each group g, so all it needs besides
        // is the last token's value at that dimension (one broadcast load per four steps), and the four lanes of a row
        // are added at the end.
        const bool tail = (M & 7) == 1 && M > 8;
        const int n_groups = tail ? M / 8 : (M + 7) / 8;     // groups that go through the tiles
        const int rows = tail ? M : 8 * n_groups;            // staged rows; rows >= M are zero
        const int n_chunks = (p.d + kMmaChunk - 1) / kMmaChunk;
        // Each warp stages its own 16 dimensions of every chunk into a ring of its own and waits only for its own
        // copies: no block-wide barrier inside the loop, so the warps drift apart and keep the fp64 pipe fed while
        // others load and widen.
        uint8_t *ring = mma_smem + (size_t)warp * Sh::kWarpRingBytes;
        // a lane copies the same pieces (row, 16-byte column) of every chunk: source pointers and ring offsets are set up once
        constexpr int kLanePieces = (kMaxCrop * Sh::kPiecesPerRow + 31) / 32;
        const T *src[kLanePieces];
        int dst_off[kLanePieces], col[kLanePieces];
#pragma unroll
        for (int i = 0; i < kLanePieces; ++i) {
            const int it = lane + 32 * i;
            const int r = it / Sh::kPiecesPerRow, c = it % Sh::kPiecesPerRow;
            col[i] = warp * kMmaWarpDims + c * Sh::kPiece;
            src[i] = r < M ? E + (size_t)tok[r] * p.d + col[i] : nullptr;     // rows M .. rows - 1 are zero-filled
            dst_off[i] = it < rows * Sh::kPiecesPerRow ? r * Sh::kWarpRowBytes + c * 16 : -1;
        }
        auto stage_chunk = [&](int ch) {
            uint8_t *dst = ring + (size_t)(ch % Sh::kStages) * Sh::kWarpStageBytes;
#pragma unroll
            for (int i = 0; i < kLanePieces; ++i) {
                if (dst_off[i] < 0) continue;
                const bool live = src[i] != nullptr && ch * kMmaChunk + col[i] < p.d;   // embed_dim is a multiple of 8: a piece is all there or not at all
                cp_async_16(dst + dst_off[i], live ? (const void *)(src[i] + (size_t)ch * kMmaChunk) : (const void *)E, live ? 16 : 0);
            }
        };
        double acc[kMmaTiles][2];
#pragma unroll
        for (int t = 0; t < kMmaTiles; ++t) acc[t][0] = acc[t][1] = 0.0;
        double tacc[4] = {0.0, 0.0, 0.0, 0.0};               // last token x groups 0..2, and its squared norm
        // the loop over the chunks, instantiated per (groups, tail) so that the multiply sequence is straight-line code
        auto gram_loop = [&](auto ng_tag, auto tail_tag) {
            constexpr int NG = decltype(ng_tag)::value;
            constexpr bool TAIL = decltype(tail_tag)::value;
            for (int s = 0; s < Sh::kStages - 1; ++s) {
                if (s < n_chunks) stage_chunk(s);
                asm volatile("cp.async.commit_group;" ::: "memory");
            }
            for (int ch = 0; ch < n_chunks; ++ch) {
                // this lane's copies of chunk ch have landed; after the warp barrier so have the other lanes', and every
                // lane is done reading the slot that the next copies overwrite
                asm volatile("cp.async.wait_group %0;" ::"n"(Sh::kStages - 2) : "memory");
                __syncwarp();
                if (ch + Sh::kStages - 1 < n_chunks) stage_chunk(ch + Sh::kStages - 1);
                asm volatile("cp.async.commit_group;" ::: "memory");
                const T *st = reinterpret_cast<const T *>(ring + (size_t)(ch % Sh::kStages) * Sh::kWarpStageBytes);
                double frag[NG][4], tv[4] = {0.0, 0.0, 0.0, 0.0};   // [group][step]
#pragma unroll
                for (int g = 0; g < NG; ++g) load_frag4(st + (g * 8 + (lane >> 2)) * kMmaWarpDims + (lane & 3) * 4, frag[g]);
                if (TAIL) load_frag4(st + (M - 1) * kMmaWarpDims + (lane & 3) * 4, tv);
#pragma unroll
                for (int step = 0; step < 4; ++step) {
#pragma unroll
                    for (int ga = 0; ga < NG; ++ga)
#pragma unroll
                        for (int gc = ga; gc < NG; ++gc) {
                            const int t = ga * 4 - ga * (ga - 1) / 2 + (gc - ga);   // constant after unrolling
                            dmma_m8n8k4(acc[t][0], acc[t][1], frag[ga][step], frag[gc][step]);
                        }
                    if (TAIL) {
#pragma unroll
                        for (int g = 0; g < NG; ++g) tacc[g] = __fma_rn(frag[g][step], tv[step], tacc[g]);
                        tacc[3] = __fma_rn(tv[step], tv[step], tacc[3]);
                    }
                }
            }
        };
        using std::integral_constant;
        switch (n_groups * 2 + (tail ? 1 : 0)) {
            case 2: gram_loop(integral_constant<int, 1>{}, integral_constant<bool, false>{}); break;
            case 3: gram_loop(integral_constant<int, 1>{}, integral_constant<bool, true>{}); break;
            case 4: gram_loop(integral_constant<int, 2>{}, integral_constant<bool, false>{}); break;
            case 5: gram_loop(integral_constant<int, 2>{}, integral_constant<bool, true>{}); break;
            case 6: gram_loop(integral_constant<int, 3>{}, integral_constant<bool, false>{}); break;
            case 7: gram_loop(integral_constant<int, 3>{}, integral_constant<bool, true>{}); break;
            default: gram_loop(integral_constant<int, 4>{}, integral_constant<bool, false>{}); break;
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        // the eight warps' partial tiles meet in shared memory (the ring is idle now)
        double *red = reinterpret_cast<double *>(mma_smem);
        {
            double *mine = red + (size_t)warp * (kMmaTiles * 64);
            int t = 0;
#pragma unroll
            for (int ga = 0; ga < 4; ++ga)
#pragma unroll
                for (int gc = ga; gc < 4; ++gc, ++t)
                    if (gc < n_groups) {
                        mine[t * 64 + (lane >> 2) * 8 + (lane & 3) * 2] = acc[t][0];
                        mine[t * 64 + (lane >> 2) * 8 + (lane & 3) * 2 + 1] = acc[t][1];
                    }
        }
        if (tail) {
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                tacc[g] += __shfl_xor_sync(0xffffffffu, tacc[g], 1);
                tacc[g] += __shfl_xor_sync(0xffffffffu, tacc[g], 2);
            }
            if ((lane & 3) == 0) {
#pragma unroll
                for (int g = 0; g < 3; ++g)
                    if (g < n_groups) tail_red[warp][g * 8 + (lane >> 2)] = tacc[g];
                if (lane == 0) tail_red[warp][M - 1] = tacc[3];
            }
        }
        __syncthreads();
        // G[a][c] for a <= c, summed over the warps in a fixed order; then the cosines
        for (int x = tid; x < M * M; x += kMmaThreads) {
            const int a = x / M, c = x % M;
            if (a > c) continue;
            if (tail && c == M - 1) {
                double g = 0.0;
                for (int w = 0; w < kMmaWarps; ++w) g += tail_red[w][a];
                S[a][c] = g;
                continue;
            }
            const int ga = a >> 3, gc = c >> 3;
            const int t = ga * 4 - ga * (ga - 1) / 2 + (gc - ga);       // index of tile (ga, gc) in the upper triangle of 4 x 4
            double g = 0.0;
            for (int w = 0; w < kMmaWarps; ++w) g += red[(size_t)w * (kMmaTiles * 64) + t * 64 + (a & 7) * 8 + (c & 7)];
            S[a][c] = g;
        }
        __syncthreads();
        if (tid < M) root[tid] = S[tid][tid] > 0.0 ? sqrt(S[tid][tid]) : 0.0;
        __syncthreads();
        for (int x = tid; x < M * M; x += kMmaThreads) {
            const int a = x / M, c = x % M;
            if (a >= c) continue;
            const double na = root[a], nc = root[c];
            const double cs = (na > 0.0 && nc > 0.0) ? S[a][c] / (na * nc) : 0.0;
            S[a][c] = cs;
            S[c][a] = cs;
        }
        __syncthreads();
    }
    if (tid < M) S[tid][tid] = 1.0;
    __syncthreads();
    // eight threads per row
    static_assert(kMmaThreads == 8 * kMaxCrop, "a row of the matrix per eight threads");
    const int a = tid >> 3;
    double mu = 0.0, var = 0.0;
    if (a < M)
        for (int c = tid & 7; c < M; c += 8) mu += S[a][c];
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) mu += __shfl_xor_sync(0xffffffffu, mu, o);
    mu /= M;
    if (a < M)
        for (int c = tid & 7; c < M; c += 8) var += (S[a][c] - mu) * (S[a][c] - mu);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) var += __shfl_xor_sync(0xffffffffu, var, o);
    if (a < M && (tid & 7) == 0) p.s_spa[tok[a]] = var / M;
}

// ---- per-frame standardisation and fusion: one CTA per frame ---------------------------------------------------
// Sums of three values over the block, the results valid in every thread.  Fixed reduction order.
__device__ __forceinline__ void block_sum3(double (&v)[3], double (*scratch)[3] /* [32] shared */) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] = warp_sum(v[i]);
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < 3; ++i) scratch[warp][i] = v[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] = 0.0;
    for (int w = 0; w < nw; ++w)
#pragma unroll
        for (int i = 0; i < 3; ++i) v[i] += scratch[w][i];
}

// Bound: latency (loads, then two reductions).  The three terms go through the two reductions (mean, variance) together
// instead of one term after the other.
__global__ void __launch_bounds__(1024) select_fuse_kernel(const SelectParams p) {
    __shared__ double scratch[2][32][3];
    const int gframe = blockIdx.x;
    const int b = find_seq(p.frame_off, p.batch, gframe);
    const int f = gframe - p.frame_off[b];
    const int n_v = p.seq_off[b + 1] - p.seq_off[b];
    const int n_frames = (n_v + p.tpf - 1) / p.tpf;
    const int nf = min(p.tpf, n_v - f * p.tpf);
    // blockDim.x >= tokens per frame (checked on the host): thread c owns grid cell c
    const int c = threadIdx.x;
    const bool valid = c < nf;
    const int j = p.seq_off[b] + f * p.tpf + c;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    double x[3] = {0.0, 0.0, 0.0};
    if (valid) {
        if (p.mask & HIPPO_SCORE_ATTN) x[0] = (double)p.attn_mass[j];
        if (p.mask & HIPPO_SCORE_SPA) x[1] = p.s_spa[j];
        if (p.mask & HIPPO_SCORE_TEMP) {
            // the previous frame always holds every cell
            const bool back = f > 0, on = f + 1 < n_frames && c < min(p.tpf, n_v - (f + 1) * p.tpf);
            double cb = back ? p.tdot[j - p.tpf] : 0.0, co = on ? p.tdot[j] : 0.0;
            if (!p.cosines) {
                const double nj = p.norm2[j], nb = back ? p.norm2[j - p.tpf] : 0.0, no = on ? p.norm2[j + p.tpf] : 0.0;
                cb = nj > 0.0 && nb > 0.0 ? cb / (sqrt(nj) * sqrt(nb)) : 0.0;
                co = nj > 0.0 && no > 0.0 ? co / (sqrt(nj) * sqrt(no)) : 0.0;
            }
            x[2] = 1.0 - (back && on ? 0.5 * (cb + co) : cb + co);
        }
    }
    double mu[3] = {x[0], x[1], x[2]}, dv[3], var[3];
    block_sum3(mu, scratch[0]);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        mu[i] /= nf;
        dv[i] = valid ? x[i] - mu[i] : 0.0;
        var[i] = dv[i] * dv[i];
    }
    block_sum3(var, scratch[1]);
    double fused = 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const unsigned bit = i == 0 ? HIPPO_SCORE_ATTN : i == 1 ? HIPPO_SCORE_SPA : HIPPO_SCORE_TEMP;
        var[i] /= nf;
        const double floor_ = 1e-24 * fmax(1.0, mu[i] * mu[i]);
        if ((p.mask & bit) && !(var[i] <= floor_)) fused += dv[i] / sqrt(var[i]);
    }
    if (valid) p.fused[j] = (float)fused;
}

// ---- top-k: one cluster of CTAs per sequence ----------------------------------------------------------------------
__device__ __forceinline__ uint32_t order_key(float x) {  // larger float -> larger key
    const uint32_t u = __float_as_uint(x);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// A sequence's keys are dealt to the CTAs of a cluster in contiguous shares, to a CTA's threads in groups of eight neighbours
// (a share of more than one round is read again per pass).  The key T of the k-th largest element comes from three histogram
// passes over its digits (11, 11 and 10 bits, top first): every CTA counts its own keys that agree with T so far, reads the
// others' counts through distributed shared memory and finds the digit by a scan of its own, which also adds up what the
// shares in front of its own hold above the digit and on it.  Then one scan of the pairs (keys > T, keys == T) gives every thread its
// first output position: the kept ones among the equal are those with the lowest indices, so position = (larger ones before) +
// min(equal ones before, equal ones to keep).
// Bound: latency (three passes of count, exchange, scan).  65,536 tokens 20 us, 160 us with one CTA and two bits per step (three
// block barriers each, keys beyond 32 per thread in shared memory); 28 us with the remote counts loaded one after the other.
constexpr int kTopByRank = 256;     // keys that are ranked by counting
constexpr int kTopThreads = 1024, kTopPerThread = 8, kTopTile = kTopThreads * kTopPerThread, kTopBins = 2048;

__global__ void __launch_bounds__(kTopThreads, 1) select_topk_kernel(const SelectParams p, const int cluster) {
    // one histogram per pass, since peers may still read the one before.  The first digit (sign, exponent, two bits) of most keys
    // falls into a few bins, so it is counted in four copies, lane modulo 4.
    __shared__ __align__(16) uint32_t copies[kTopBins * 4];
    __shared__ uint32_t hist1[kTopBins], hist2[kTopBins / 2];
    uint32_t *hist0 = copies;
    __shared__ uint32_t wsum[32], s_digit, s_above;
    __shared__ uint32_t wlow[32];
    __shared__ unsigned long long w64[32], s_lower;
    const int b = blockIdx.x / cluster, rank = blockIdx.x % cluster, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = p.seq_off[b + 1] - p.seq_off[b], k = p.k[b];
    for (int i = tid; i < kTopBins; i += kTopThreads) { reinterpret_cast<uint4 *>(hist0)[i] = make_uint4(0, 0, 0, 0); hist1[i] = 0; }
    hist2[tid] = 0;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const float *score = p.fused + p.seq_off[b];
    int32_t *out = p.kept + p.k_off[b];
    if (k <= 0) return;                           // the same for the whole cluster
    if (n <= kTopByRank) {
        // A key's rank is the number of better ones; several threads per key look at every kParts-th of the others.  Two barriers where
        // the digits take a dozen.
        if (rank > 0) return;
        constexpr int kParts = kTopThreads / kTopByRank;
        uint32_t *keys = hist2, *kept = hist1;
        if (tid < n) keys[tid] = order_key(score[tid]);
        __syncthreads();
        const int i = tid / kParts;
        const uint32_t mine = i < n ? keys[i] : 0u;
        int better = 0, j = tid % kParts;
        for (; j < min(i, n); j += kParts) better += keys[j] >= mine ? 1 : 0;           // an equal key in front is better
        if (j == i) j += kParts;
        for (; j < n; j += kParts) better += keys[j] > mine ? 1 : 0;
#pragma unroll
        for (int o = 1; o < kParts; o <<= 1) better += __shfl_xor_sync(0xffffffffu, better, o);
        const bool keep = i < n && better < k;
        const unsigned bits = __ballot_sync(0xffffffffu, keep && tid % kParts == 0);
        if (lane == 0) kept[warp] = __popc(bits);
        __syncthreads();
        const int before = (int)__reduce_add_sync(0xffffffffu, lane < warp ? kept[lane] : 0u) + __popc(bits & ((1u << lane) - 1));
        if (keep && tid % kParts == 0) out[before] = i;
        return;
    }
    const int begin = (int)((long long)n * rank / cluster), end = (int)((long long)n * (rank + 1) / cluster);
    const int rounds = (end - begin + kTopTile - 1) / kTopTile;
    uint32_t key[kTopPerThread];
    auto load = [&](int round) {
#pragma unroll
        for (int e = 0; e < kTopPerThread; ++e) {
            const int i = begin + round * kTopTile + tid * kTopPerThread + e;
            key[e] = i < end ? order_key(score[i]) : 0u;
        }
    };
    auto live = [&](int round, int e) { return begin + round * kTopTile + tid * kTopPerThread + e < end; };
    load(0);
    __syncthreads();
    uint32_t T = 0, mask = 0;
    unsigned long long base = 0;                  // (larger than T) << 32 | (equal to T) in the shares in front of this CTA's
    int need = k;                                 // the wanted element is the need-th largest among the keys that agree with T so far
    auto find_digit = [&](auto pass_tag) {
        constexpr int pass = decltype(pass_tag)::value, shift = pass == 0 ? 21 : pass == 1 ? 10 : 0;
        constexpr uint32_t digits = pass == 2 ? 1023u : 2047u;
        for (int r = 0; r < rounds; ++r) {
            if (rounds > 1) load(r);
#pragma unroll
            for (int e = 0; e < kTopPerThread; ++e)
                if (live(r, e) && (key[e] & mask) == T) {
                    const uint32_t bin = (key[e] >> shift) & digits;
                    atomicAdd(pass == 0 ? &hist0[bin * 4 + (lane & 3)] : pass == 1 ? &hist1[bin] : &hist2[bin], 1u);
                }
        }
        if (pass == 0) {
            __syncthreads();
            const uint4 v0 = reinterpret_cast<const uint4 *>(copies)[2 * tid], v1 = reinterpret_cast<const uint4 *>(copies)[2 * tid + 1];
            __syncthreads();                      // folded in place
            hist0[2 * tid] = (v0.x + v0.y) + (v0.z + v0.w);
            hist0[2 * tid + 1] = (v1.x + v1.y) + (v1.z + v1.w);
        }
        if (cluster > 1) cluster_sync_all(); else __syncthreads();
        // counts over the cluster and their sums from the top: thread t owns the bins 2 t, 2 t + 1 counted from the top
        constexpr int kBins = pass == 2 ? kTopBins / 2 : kTopBins;
        uint32_t c[2], low[2] = {0, 0}, w[2][7];   // low: in the shares in front of this CTA's
#pragma unroll
        for (int h = 0; h < 2; ++h) {             // every remote load is in flight before the first is used
            const int bin = kBins - 1 - (2 * tid + h);
            c[h] = bin < 0 ? 0u : pass == 0 ? hist0[bin] : pass == 1 ? hist1[bin] : hist2[bin];
#pragma unroll
            for (int q = 1; q < 8; ++q) {
                w[h][q - 1] = 0;
                if (bin >= 0 && q < cluster)
                    w[h][q - 1] = ld_cluster_u32(cluster_map(smem_u32(pass == 0 ? &hist0[bin] : pass == 1 ? &hist1[bin] : &hist2[bin]), (uint32_t)(rank ^ q)));
            }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int q = 0; q < 7; ++q) {
                c[h] += w[h][q];
                low[h] += (rank ^ (q + 1)) < rank ? w[h][q] : 0u;
            }
        // keys in higher bins, of all shares and (in a cluster) of those in front
        auto scan = [&](uint32_t mine, uint32_t *sums) {
            uint32_t inc = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) { const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += v; }
            if (lane == 31) sums[warp] = inc;
            return inc - mine;
        };
        auto in_front = [&](const uint32_t *sums) { return __reduce_add_sync(0xffffffffu, lane < warp ? sums[lane] : 0u); };
        uint32_t before = scan(c[0] + c[1], wsum), lower = cluster > 1 ? scan(low[0] + low[1], wlow) : 0u;
        __syncthreads();
        before += in_front(wsum);
        if (cluster > 1) lower += in_front(wlow);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (before < (uint32_t)need && (uint32_t)need <= before + c[h]) {
                s_digit = (uint32_t)(kBins - 1 - (2 * tid + h));
                s_above = before;
                s_lower = (unsigned long long)lower << 32 | low[h];
            }
            before += c[h];
            lower += low[h];
        }
        __syncthreads();
        T |= s_digit << shift;
        mask |= digits << shift;
        need -= (int)s_above;                     // after the last pass: elements equal to T to keep
        // what the shares in front of this one have above the digit, and, should it be the last one, on it
        base = (base & 0xffffffff00000000ull) + s_lower;
    };
    find_digit(std::integral_constant<int, 0>{});
    find_digit(std::integral_constant<int, 1>{});
    find_digit(std::integral_constant<int, 2>{});
    unsigned long long run = base;
    for (int r = 0; r < rounds; ++r) {
        if (rounds > 1) load(r);
        unsigned long long mine = 0;
#pragma unroll
        for (int e = 0; e < kTopPerThread; ++e)
            if (live(r, e)) mine += key[e] > T ? 1ull << 32 : key[e] == T ? 1ull : 0ull;
        unsigned long long inc = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const unsigned long long v = __shfl_up_sync(0xffffffffu, inc, o); if (lane >= o) inc += v; }
        __syncthreads();                          // w64 of the round before has been read
        if (lane == 31) w64[warp] = inc;
        __syncthreads();
        unsigned long long sums = w64[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const unsigned long long v = __shfl_up_sync(0xffffffffu, sums, o); if (lane >= o) sums += v; }
        const unsigned long long in_front = __shfl_sync(0xffffffffu, sums, warp ? warp - 1 : 0);
        const unsigned long long at = run + (warp ? in_front : 0ull) + inc - mine;
        run += __shfl_sync(0xffffffffu, sums, 31);
        uint32_t gt = (uint32_t)(at >> 32), eq = (uint32_t)at;
#pragma unroll
        for (int e = 0; e < kTopPerThread; ++e) {
            if (!live(r, e)) continue;
            const bool g = key[e] > T, q = key[e] == T;
            if (g || (q && eq < (uint32_t)need)) out[gt + min(eq, (uint32_t)need)] = begin + r * kTopTile + tid * kTopPerThread + e;
            gt += g; eq += q;
        }
    }
    if (cluster > 1) cluster_sync_all();          // nobody leaves while its shared memory may be read
}

// ---- uniform budget per frame ------------------------------------------------------------------------------------
// Budgets of one sequence, by one thread: floor(k / F) per frame, the first k mod F frames one more; a frame with fewer
// tokens than its budget keeps them all and the shortfall goes, one token at a time in frame order, to the frames that
// still have room.  Also the first output position of every frame.
__global__ void select_budget_kernel(const SelectParams p) {
    const int b = blockIdx.x;
    if (threadIdx.x != 0) return;
    const int n = p.seq_off[b + 1] - p.seq_off[b], k = p.k[b];
    const int F = (n + p.tpf - 1) / p.tpf;
    int *budget = p.frame_budget + p.frame_off[b], *first = p.frame_out + p.frame_off[b];
    int given = 0;
    for (int f = 0; f < F; ++f) {
        const int want = k / F + (f < k % F ? 1 : 0), have = min(p.tpf, n - f * p.tpf);
        budget[f] = min(want, have);
        given += budget[f];
    }
    while (given < k)
        for (int f = 0; f < F && given < k; ++f)
            if (budget[f] < min(p.tpf, n - f * p.tpf)) { ++budget[f]; ++given; }
    int acc = 0;
    for (int f = 0; f < F; ++f) { first[f] = acc; acc += budget[f]; }
}

// One CTA per frame, thread c owns grid cell c: its rank among the frame's tokens by (score as fp32 descending, index
// ascending) is a count over the frame's keys in shared memory; the kept ones are written in index order.
__global__ void __launch_bounds__(1024) select_frame_topk_kernel(const SelectParams p) {
    __shared__ uint32_t keys[1024];
    __shared__ int warp_cnt[32];
    const int gframe = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = find_seq(p.frame_off, p.batch, gframe);
    const int f = gframe - p.frame_off[b];
    const int n_v = p.seq_off[b + 1] - p.seq_off[b];
    const int nf = min(p.tpf, n_v - f * p.tpf);
    const int kf = p.frame_budget[gframe];
    const bool valid = tid < nf;
    const uint32_t key = valid ? order_key(p.fused[p.seq_off[b] + f * p.tpf + tid]) : 0u;
    keys[tid] = key;
    __syncthreads();
    int rank = 0;
    for (int c = 0; c < nf; ++c) {
        const uint32_t other = keys[c];
        rank += (other > key || (other == key && c < tid)) ? 1 : 0;
    }
    const bool sel = valid && rank < kf;
    const unsigned bal = __ballot_sync(0xffffffffu, sel);
    if (lane == 0) warp_cnt[warp] = __popc(bal);
    __syncthreads();
    int before = __popc(bal & ((1u << lane) - 1));
    for (int w = 0; w < warp; ++w) before += warp_cnt[w];
    if (sel) p.kept[p.k_off[b] + p.frame_out[gframe] + before] = f * p.tpf + tid;
}

// ---- whole frames at a regular stride --------------------------------------------------------------------------------
// Output position i of sequence b: with m = ceil(k / T) frames kept out of the Fc complete ones, frame floor(q * Fc / m)
// for q = i / T, cell i mod T (the last kept frame is cut short when k is not a multiple of T); when k reaches Fc * T, or
// there is no complete frame, the first k tokens.
__global__ void select_frames_kernel(const SelectParams p) {
    const int b = blockIdx.y;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = p.k[b];
    if (i >= k) return;
    const int n = p.seq_off[b + 1] - p.seq_off[b], T = p.tpf, Fc = n / T;
    int idx = i;
    if (Fc > 0 && (long long)k < (long long)Fc * T) {
        const int m = (k + T - 1) / T;
        idx = (int)((long long)(i / T) * Fc / m) * T + i % T;
    }
    p.kept[p.k_off[b] + i] = idx;
}

__global__ void select_copy_keys_kernel(const float *keys, float *fused, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) fused[i] = keys[i];
}

// A kernel that begins with griddepcontrol.wait: its launch overlaps the end of its predecessor in the stream.
template <typename... Args>
static cudaError_t launch_dependent(void (*kernel)(Args...), long long grid, int threads, int cluster, size_t smem, cudaStream_t s, Args... args) {
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)cluster;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

struct SelectWs { size_t norm2_off, tdot_off, spa_off, budget_off, total; };
static SelectWs select_ws(long long total_tokens, long long total_frames) {
    SelectWs w;
    const size_t a = align_up((size_t)total_tokens * sizeof(double), 256);
    w.norm2_off = kWsHeaderBytes;
    w.tdot_off = w.norm2_off + a;
    w.spa_off = w.tdot_off + a;
    w.budget_off = w.spa_off + a;       // per-frame policy: budget and first output position of every frame
    w.total = w.budget_off + align_up((size_t)total_frames * 2 * sizeof(int), 256);
    return w;
}

}  // namespace hippo

extern "C" {

size_t hippo_select_workspace_bytes(int32_t batch, const int32_t *n_visual, int32_t grid_h, int32_t grid_w,
                                    int32_t crop_h, int32_t crop_w) {
    (void)crop_h; (void)crop_w;
    if (batch <= 0 || !n_visual || grid_h <= 0 || grid_w <= 0) return 0;
    long long t = 0, f = 0;
    const long long tpf = (long long)grid_h * grid_w;
    for (int b = 0; b < batch; ++b) { if (n_visual[b] <= 0) return 0; t += n_visual[b]; f += (n_visual[b] + tpf - 1) / tpf; }
    return hippo::select_ws(t, f).total;
}

int32_t hippo_select_tokens(int32_t batch, const int32_t *n_visual, int32_t grid_h, int32_t grid_w, int32_t crop_h,
                            int32_t crop_w, int32_t embed_dim, int32_t dtype, const void *embeds,
                            const float *attn_mass, const int32_t *k, const int32_t *kept_offsets,
                            uint32_t score_mask, int32_t *kept_idx, float *fused_score, void *workspace,
                            size_t workspace_bytes, void *stream) {
    return hippo_select_tokens_policy(batch, n_visual, grid_h, grid_w, crop_h, crop_w, embed_dim, dtype, embeds, attn_mass, k,
                                      kept_offsets, score_mask, HIPPO_SELECT_HOLISTIC, nullptr, kept_idx, fused_score,
                                      workspace, workspace_bytes, stream);
}

int32_t hippo_select_tokens_policy(int32_t batch, const int32_t *n_visual, int32_t grid_h, int32_t grid_w, int32_t crop_h,
                                   int32_t crop_w, int32_t embed_dim, int32_t dtype, const void *embeds,
                                   const float *attn_mass, const int32_t *k, const int32_t *kept_offsets,
                                   uint32_t score_mask, int32_t policy, const float *random_keys, int32_t *kept_idx,
                                   float *fused_score, void *workspace, size_t workspace_bytes, void *stream) {
    using namespace hippo;
    const char *who = "hippo_select_tokens";
    if (batch <= 0 || !n_visual || !k) return fail(HIPPO_ERR_INVALID_ARG, "%s: bad batch / null host arrays", who);
    if (policy < HIPPO_SELECT_HOLISTIC || policy > HIPPO_SELECT_FRAMES) return fail(HIPPO_ERR_INVALID_ARG, "%s: unknown policy %d", who, policy);
    const bool scored = policy == HIPPO_SELECT_HOLISTIC || policy == HIPPO_SELECT_UNIFORM_PER_FRAME;
    if (policy == HIPPO_SELECT_RANDOM && !random_keys) return fail(HIPPO_ERR_INVALID_ARG, "%s: the random policy needs random_keys", who);
    if (batch > kSelMaxBatch) return fail(HIPPO_ERR_UNSUPPORTED_SHAPE, "%s: batch > %d", who, kSelMaxBatch);
    if (grid_h <= 0 || grid_w <= 0 || crop_h <= 0 || crop_w <= 0 || embed_dim <= 0)
        return fail(HIPPO_ERR_INVALID_ARG, "%s: non-positive geometry", who);
    if (dtype != HIPPO_DTYPE_FP32 && dtype != HIPPO_DTYPE_BF16) return fail(HIPPO_ERR_INVALID_ARG, "%s: unknown dtype", who);
    if (crop_h * crop_w > kMaxCrop) return fail(HIPPO_ERR_UNSUPPORTED_SHAPE, "%s: crop larger than %d tokens", who, kMaxCrop);
    if ((long long)grid_h * grid_w > 1024) return fail(HIPPO_ERR_UNSUPPORTED_SHAPE, "%s: more than 1024 tokens per frame", who);
    if (embed_dim % 8) return fail(HIPPO_ERR_UNSUPPORTED_SHAPE, "%s: embed_dim must be a multiple of 8", who);
    if (!workspace || (scored && (!embeds || !attn_mass)) || (policy != HIPPO_SELECT_FRAMES && !fused_score))
        return fail(HIPPO_ERR_INVALID_ARG, "%s: null pointer", who);
    if ((score_mask & ~HIPPO_SCORE_ALL) != 0) return fail(HIPPO_ERR_INVALID_ARG, "%s: unknown score_mask bits", who);
    if ((uintptr_t)workspace & 255) return fail(HIPPO_ERR_INVALID_ARG, "%s: workspace must be 256-byte aligned", who);
    if (scored && ((uintptr_t)embeds & 15)) return fail(HIPPO_ERR_INVALID_ARG, "%s: embeds must be 16-byte aligned", who);

    SelectParams p;
    p.tpf = grid_h * grid_w;
    long long tok = 0, frames = 0, ksum = 0;
    for (int b = 0; b < batch; ++b) {
        if (n_visual[b] <= 0) return fail(HIPPO_ERR_INVALID_ARG, "%s: n_visual[%d] <= 0", who, b);
        if (k[b] < 0 || k[b] > n_visual[b]) return fail(HIPPO_ERR_INVALID_ARG, "%s: k[%d] outside [0, n_visual]", who, b);
        p.seq_off[b] = (int)tok; p.frame_off[b] = (int)frames; p.k[b] = k[b];
        if (kept_offsets && kept_offsets[b] < 0) return fail(HIPPO_ERR_INVALID_ARG, "%s: kept_offsets[%d] < 0", who, b);
        p.k_off[b] = kept_offsets ? kept_offsets[b] : (int)ksum;
        tok += n_visual[b]; frames += (n_visual[b] + p.tpf - 1) / p.tpf; ksum += k[b];
        if (tok > 0x7fffffffLL / 2) return fail(HIPPO_ERR_UNSUPPORTED_SHAPE, "%s: too many tokens", who);
    }
    p.seq_off[batch] = (int)tok; p.frame_off[batch] = (int)frames; p.k_off[batch] = (int)ksum;
    if (ksum > 0 && !kept_idx) return fail(HIPPO_ERR_INVALID_ARG, "%s: null kept_idx", who);
    SelectWs w = select_ws(tok, frames);
    if (workspace_bytes < w.total) return fail(HIPPO_ERR_WORKSPACE_TOO_SMALL, "%s: workspace %zu < %zu bytes", who, workspace_bytes, w.total);
    p.embeds = embeds; p.attn_mass = attn_mass; p.fused = fused_score; p.kept = kept_idx;
    p.norm2 = (double *)((char *)workspace + w.norm2_off);
    p.tdot = (double *)((char *)workspace + w.tdot_off);
    p.s_spa = (double *)((char *)workspace + w.spa_off);
    p.frame_budget = (int *)((char *)workspace + w.budget_off);
    p.frame_out = p.frame_budget + frames;
    p.batch = batch; p.grid_h = grid_h; p.grid_w = grid_w; p.crop_h = crop_h; p.crop_w = crop_w; p.d = embed_dim;
    p.crops_y = ceil_div(grid_h, crop_h); p.crops_x = ceil_div(grid_w, crop_w);
    p.mask = score_mask;
    cudaStream_t s = (cudaStream_t)stream;
    if (policy == HIPPO_SELECT_FRAMES) {
        // an index rule: no scores are formed, fused_score is not written
        int kmax = 0;
        for (int b = 0; b < batch; ++b) kmax = k[b] > kmax ? k[b] : kmax;
        if (kmax > 0) {
            select_frames_kernel<<<dim3((unsigned)ceil_div(kmax, 256), (unsigned)batch), 256, 0, s>>>(p);
            count_launches(1);
        }
        HIPPO_CUDA_TRY(cudaGetLastError());
        return HIPPO_OK;
    }
    if (policy == HIPPO_SELECT_RANDOM) {
        // the caller's keys take the place of the fused score (and are returned as such)
        select_copy_keys_kernel<<<(unsigned)((tok + 255) / 256), 256, 0, s>>>(random_keys, fused_score, (int)tok);
        count_launches(1);
    }
    const bool need_emb = scored && (score_mask & (HIPPO_SCORE_TEMP | HIPPO_SCORE_SPA)) != 0;
    // Without the spatial term only norms and products with the next frame are needed, which is one pass of select_dots_kernel
    // (32,768 of 4,096: 105 us against 196 for the tiles).  bf16 otherwise: the integer tensor path, except where its fixed cost
    // (set-up, merge and scores of a tile) outweighs the shorter loop - whole selection, integer path against fp64 kernels: 2,000
    // tokens of 2,048 44.9 / 37.6 us, 1,000 of 3,584 45.9 / 45.4, 512 of 8,192 54 / 70, 3,000 of 4,096 55 / 68, 32,768 of 4,096 195 /
    // 290, 65,536 of 8,192 552 / 917 - and where its tiles of 128 rows hold a few tokens each: many crops, few frames (one frame of
    // 32 x 32, crops of one token, 4,096 dimensions: 388 / 55; four sequences of 750 in such a grid 115 / 98).  The fp64 kernels take
    // about 10 us, the longer of a crop's own chain (3.4 to 12.5 ns per dimension, by its size) and their share of
    // the fp64 rate (2.2 ps per element), and half of the other.  4,884 tokens of 2,872, 6,628 of 1,384, 14,950 of 1,216: 54.5 / 82,
    // 44 / 59, 73 / 86.
    bool gram = dtype == HIPPO_DTYPE_BF16 && (score_mask & HIPPO_SCORE_SPA) && embed_dim <= kGramMaxDim &&
                (embed_dim >= 4096 || tok * embed_dim >= 5000000);
    if (need_emb && gram) {
        double tiles_us = 0.0;
        const int32_t rc = select_gram_cost(p, tiles_us);
        if (rc != HIPPO_OK) return rc;
        int area = 0;                 // tokens of the fullest crop
        for (int b = 0; b < batch; ++b) {
            int first = 0;
            for (int y = 0; y < crop_h && y < grid_h; ++y) {
                const int left = n_visual[b] - y * grid_w, w = crop_w < grid_w ? crop_w : grid_w;
                first += left < 0 ? 0 : left < w ? left : w;
            }
            area = first > area ? first : area;
        }
        const double ns_per_dim[5] = {0.0, 3.4, 4.5, 10.2, 12.5};            // by groups of eight tokens in a crop
        const double chain_us = area > 1 ? 1e-3 * ns_per_dim[(area + 6) / 8] * embed_dim : 0.0, rate_us = 2.2e-6 * tok * embed_dim;
        gram = tiles_us < 10.0 + (chain_us > rate_us ? chain_us + 0.5 * rate_us : rate_us + 0.5 * chain_us);
    }
    p.cosines = need_emb && gram ? 1 : 0;
    if (need_emb && gram) {
        const int32_t rc = launch_select_gram(p, (WsHeader *)workspace, s);
        if (rc != HIPPO_OK) return rc;
    } else if (need_emb) {
        // norms and next-frame products, and in front of them the crops where the mask has the spatial term
        const bool spa = (score_mask & HIPPO_SCORE_SPA) != 0, fp32 = dtype == HIPPO_DTYPE_FP32;
        const int dots = ceil_div((int)tok, kDotsThreads / 32);
        if (spa) {
            static PerDeviceOnce spa_attr;
            int dev;
            if (spa_attr.needed(dev)) {
                HIPPO_CUDA_TRY(cudaFuncSetAttribute(select_spatial_mma_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MmaShape<float>::kSmemBytes));
                HIPPO_CUDA_TRY(cudaFuncSetAttribute(select_spatial_mma_kernel<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MmaShape<__nv_bfloat16>::kSmemBytes));
                spa_attr.mark(dev);
            }
            const long long grid = frames * p.crops_y * p.crops_x + dots;
            HIPPO_CUDA_TRY(fp32 ? launch_dependent(select_spatial_mma_kernel<float>, grid, kMmaThreads, 1, MmaShape<float>::kSmemBytes, s, p)
                                : launch_dependent(select_spatial_mma_kernel<__nv_bfloat16>, grid, kMmaThreads, 1, MmaShape<__nv_bfloat16>::kSmemBytes, s, p));
        } else {
            HIPPO_CUDA_TRY(fp32 ? launch_dependent(select_dots_kernel<float>, dots, kDotsThreads, 1, 0, s, p)
                                : launch_dependent(select_dots_kernel<__nv_bfloat16>, dots, kDotsThreads, 1, 0, s, p));
        }
        count_launches(1);
    }
    const int fuse_threads = ((p.tpf + 31) / 32) * 32;
    if (scored) {
        HIPPO_CUDA_TRY(launch_dependent(select_fuse_kernel, frames, fuse_threads, 1, 0, s, p));
        count_launches(1);
    }
    if (ksum > 0 && policy == HIPPO_SELECT_UNIFORM_PER_FRAME) {
        select_budget_kernel<<<batch, 32, 0, s>>>(p);
        select_frame_topk_kernel<<<(unsigned)frames, fuse_threads, 0, s>>>(p);
        count_launches(2);
    } else if (ksum > 0) {
        // half of the threads' key registers in use: 8 CTAs from 16k tokens on
        int longest = 0;
        for (int b = 0; b < batch; ++b) longest = n_visual[b] > longest ? n_visual[b] : longest;
        int cluster = 1;
        while (cluster < 8 && longest > cluster * kTopTile / 2) cluster *= 2;
        HIPPO_CUDA_TRY(launch_dependent(select_topk_kernel, batch * cluster, kTopThreads, cluster, 0, s, p, cluster));
        count_launches(1);
    }
    HIPPO_CUDA_TRY(cudaGetLastError());
    return HIPPO_OK;
}

}  // extern "C"
