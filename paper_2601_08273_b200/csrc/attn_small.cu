// Low-latency split-KV attention for few packed rows over a short cache: the draft model's decode step over the
// pruned KV (Section 3.2, drafting phase: one or two query tokens, R = q_len * G <= 16 packed rows, some hundred to some
// thousand keys).  Such a call moves a megabyte or two, so its cost is the length of the dependency chain, not bandwidth:
// one launch, operands go from global memory straight into the registers the tensor instruction reads them from, and
// every load of a step is in flight before the first one is used.
//
// One thread-block cluster per (sequence, kv head) unit; the 32-key blocks of the unit's cache are dealt to the warps of
// the cluster.  A warp does, per block of 32 keys, with mma.sync m16n8k16 (bf16 in, fp32 accumulate):
//   scores  S[16 rows x 8 keys] = Q K^T.  The contraction index may be permuted as long as both operands agree, so lane
//           (g, t) = (lane / 4, lane % 4) holds, of key g of a group of eight, the dimensions j*32 + t*8 .. + 7: plain
//           16-byte loads, 64 contiguous bytes per key and load.
//   softmax running row maxima per warp (two shuffles); the accumulator layout of S (row g, keys 2t, 2t + 1) is the
//           layout of the second contraction's B operand, so probabilities never leave their registers.
//   output  O^T[16 dims x 8 rows] += V^T P^T.  Lane (g, t) loads dimensions 8g .. 8g + 7 of keys 2t, 2t + 1, 2t + 8,
//           2t + 9 of a group of sixteen (whole rows per load) and interleaves pairs of keys with byte permutes; the
//           order of the output dimensions inside the instruction is free, so a lane ends with 8 neighbouring ones.
// Probabilities are fp32: each is split into three bf16 terms (8 + 8 + 8 significant bits), three instructions per tile.
// tcgen05 is not used: its 128 x N tile has one row block too many here and costs a tensor-memory allocation, barriers
// and a descriptor round trip per call, which is most of the time this kernel takes in total.
//
// Bound by latency: two dependent round trips to memory (lengths and page ids, then keys and values; one for an
// identity-mapped cache), the softmax and the merge.  Measured per call in a chain of 28 layers: 758 keys (0.39 MB) 3.5 us, 5.8 us
// with the CUDA-core kernel that stood here before; 3,537 keys (1.8 MB, from HBM) 4.3 us, 10.5 us through tensor memory.
//
// The warps of a CTA merge through shared memory.  Row r of the unit is merged by CTA r mod cluster size: every CTA
// pushes its (m, l, O[r]) into that CTA's shared memory with remote stores, and after a cluster barrier the owners
// merge what they received and write the output.  An earlier barrier, entered at the start and waited for before the push,
// tells that every CTA of the cluster is running.
#include <math.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace hippo {

constexpr int kSmBlock = 32;            // keys a warp takes at a time
constexpr int kSmMaxWarps = 16;
constexpr int kSmMaxCluster = 16;
constexpr int kSmMaxRows = 16;
constexpr float kSmLog2e = 1.4426950408889634f;
constexpr float kSmLn2 = 0.6931471805599453f;

__device__ __forceinline__ void sm_st_cluster_v2(uint32_t addr, float a, float b) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(a), "f"(b) : "memory");
}
__device__ __forceinline__ void sm_st_cluster_v4(uint32_t addr, float4 v) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ uint4 sm_ldg(const __nv_bfloat16 *p) { return __ldg(reinterpret_cast<const uint4 *>(p)); }
// with an L2 eviction policy
__device__ __forceinline__ uint4 sm_ldg_hint(const __nv_bfloat16 *p, uint64_t pol) {
    uint4 v;
    asm("ld.global.nc.L2::cache_hint.v4.b32 {%0, %1, %2, %3}, [%4], %5;" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(pol));
    return v;
}
// a word that another kernel may be writing: from L2, so that no old line stays in L1
__device__ __forceinline__ int sm_peek(const int32_t *p) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void sm_mma(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t sm_pack(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// (x, y) as three bf16 pairs whose sums are x and y to fp32 precision
__device__ __forceinline__ void sm_split3(float x, float y, uint32_t (&w)[3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        w[i] = sm_pack(x, y);
        x -= __uint_as_float(w[i] << 16);
        y -= __uint_as_float(w[i] & 0xffff0000u);
    }
}

// Shared memory: warps' partials m[W][16] | l[W][16] | O[W][16 or 8 rows][D + 4], then what the cluster peers push:
// (m, l)[32] | O[32][D].  A row's partials take an entry each: entry = (r / cluster size) * cluster size + peer < 32.
template <int D, int NT>
struct SmallSmem {
    static constexpr int kRows = 8 * NT;
    static constexpr int kOStride = D + 4;
    static constexpr int kEntries = 2 * kSmMaxCluster;
    __host__ __device__ static constexpr int ml_off() { return 0; }
    __host__ __device__ static constexpr int o_off(int warps) { return 2 * warps * kRows; }
    __host__ __device__ static constexpr int recv_ml_off(int warps) { return o_off(warps) + warps * kRows * kOStride; }
    __host__ __device__ static constexpr int recv_o_off(int warps) { return recv_ml_off(warps) + 2 * kEntries; }
    __host__ __device__ static constexpr size_t bytes(int warps) { return 4 * (size_t)(recv_o_off(warps) + kEntries * D); }
};

// The warp's partial outputs again, for the entries that came out NaN.  With an infinite value the three terms of a probability are no
// longer their sum (0 * inf, inf - inf): here every product is formed with the fp32 probability, so a visible infinite value is
// infinite in the output, and what is NaN by the definition (a masked key's 0 * inf among it) stays NaN.  Out of line and slow:
// only a warp that has found a NaN comes here.
template <int D, int NT>
__device__ __noinline__ void attn_small_redo(const AttnParams &p, int b, int hk, int first, int stride, int kvl, const float *m_warp, float *o_warp) {
    const int lane = threadIdx.x & 31, G = p.group;
    const __nv_bfloat16 *kp = (const __nv_bfloat16 *)p.k_pages, *vp = (const __nv_bfloat16 *)p.v_pages;
    for (int r = 0; r < p.rows; ++r) {
        const __nv_bfloat16 *q = (const __nv_bfloat16 *)p.q + (((size_t)b * p.q_len + r / G) * p.n_q_heads + hk * G + r % G) * D;
        const float ref = m_warp[r] == -INFINITY ? 0.f : m_warp[r];
        float acc[D / 32];
        for (int c = 0; c < D / 32; ++c) acc[c] = 0.f;
        for (int blk = first; blk * kSmBlock < kvl; blk += stride) {
            const int pid = page_of(p.page_table, p.max_pages_per_seq, b, blk / (kPageSize / kSmBlock));
            const size_t base = (((size_t)pid * p.n_kv_heads + hk) * kPageSize + (blk % (kPageSize / kSmBlock)) * kSmBlock) * D;
            const int key = blk * kSmBlock + lane, live = min(kSmBlock, kvl - blk * kSmBlock);
            float w = 0.f;
            if (lane < live && key <= kvl - p.q_len + r / G) {
#pragma unroll 1
                for (int d = 0; d < D; ++d) w = fmaf(__bfloat162float(q[d]), __bfloat162float(kp[base + lane * D + d]), w);
                w = ex2_approx(w * p.scale * kSmLog2e - ref);
            }
#pragma unroll 1
            for (int j = 0; j < live; ++j) {
                const float wj = __shfl_sync(0xffffffffu, w, j);
                for (int c = 0; c < D / 32; ++c) acc[c] = fmaf(wj, __bfloat162float(vp[base + j * D + c * 32 + lane]), acc[c]);
            }
        }
        for (int c = 0; c < D / 32; ++c) {
            float *o = o_warp + r * SmallSmem<D, NT>::kOStride + c * 32 + lane;
            if (isnan(*o)) *o = acc[c];
        }
    }
}

// The draft's pruned cache is read again by every token: kept in L2 beside a verification pass that streams through it (28 layers hold 11 MB
// of 126 at 758 keys, 51 at the 32k step's 3,537; beside 104 SMs of verification that step takes 1,425 us with either policy).
__device__ __forceinline__ uint64_t small_policy(const AttnParams &p) { return p.kv_resident ? l2_policy_evict_last() : l2_policy_evict_first(); }

// Ahead of the wait for the predecessor in the stream: asks L2 for what the warp is going to read.  These are hints and nothing else: a
// line that the predecessor writes later is current in L2 all the same, and the values used here (length, page ids) are looked up again
// after the wait.  They may be stale or not yet written, so they count only inside their bounds.  us per call in a chain of 28, cold
// caches: 758 keys 4.0 -> 3.9, 3,537 keys 4.9 -> 4.3, 33,000 keys 13.7 -> 11.7, eight sequences of 2,000 keys 8.1 -> 6.6.
template <int D>
__device__ __forceinline__ void sm_prefetch(const AttnParams &p, int b, int hk, int first, int stride, bool queries, int max_blocks, uint64_t pol) {
    const int lane = threadIdx.x & 31;
    if (queries && lane < p.q_len) {
        const __nv_bfloat16 *q = (const __nv_bfloat16 *)p.q + (((size_t)b * p.q_len + lane) * p.n_q_heads + hk * p.group) * D;
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(q), "r"((uint32_t)(p.group * D * 2)) : "memory");
    }
    // the first step's blocks; later ones, and those behind a page table, only as far as the length is known to reach
    const int blk = first + (lane >> 1) * stride;
    if (blk >= max_blocks) return;
    int pid = b * p.max_pages_per_seq + blk / (kPageSize / kSmBlock);
    if (p.page_table || blk != first) {
        if (p.kv_len && blk * kSmBlock >= sm_peek(p.kv_len + b)) return;
        if (p.page_table) pid = sm_peek(p.page_table + (size_t)b * p.max_pages_per_seq + blk / (kPageSize / kSmBlock));
    }
    if ((unsigned)pid >= (unsigned)p.n_pages) return;
    const __nv_bfloat16 *src = (const __nv_bfloat16 *)(lane & 1 ? p.v_pages : p.k_pages) +
                               (((size_t)pid * p.n_kv_heads + hk) * kPageSize + (blk % (kPageSize / kSmBlock)) * kSmBlock) * D;
    asm volatile("cp.async.bulk.prefetch.L2.global.L2::cache_hint [%0], %1, %2;" ::"l"(src), "r"((uint32_t)(kSmBlock * D * 2)), "l"(pol) : "memory");
}

template <int D, int NT, bool kPrefetch>   // head size; groups of eight packed rows; see small_prefetch
__global__ void __launch_bounds__(D == 64 ? 512 : 256) attn_small_kernel(const __grid_constant__ AttnParams p, const int cluster_size) {
    using S = SmallSmem<D, NT>;
    constexpr int kKV4 = D / 32;          // 16-byte loads of a lane per key of the score operand
    constexpr int kDT = D / 16;           // 16-dimension tiles of the output
    extern __shared__ __align__(16) float smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int W = blockDim.x >> 5;
    const int R = p.rows, G = p.group, Hkv = p.n_kv_heads;
    const int unit = blockIdx.x / cluster_size, rank = blockIdx.x % cluster_size;
    const int b = unit / Hkv, hk = unit % Hkv;
    const __nv_bfloat16 *kp = (const __nv_bfloat16 *)p.k_pages, *vp = (const __nv_bfloat16 *)p.v_pages;
    const int stride = W * cluster_size;                        // blocks of 32 keys from one step of this warp to the next
    const int first = warp * cluster_size + rank;
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");     // this CTA runs: its peers may push into its memory
    const int max_blocks = (p.max_kv_len + kSmBlock - 1) / kSmBlock;
    // Where the policy and the query rows are worked out decides the order that the compiler gives a step's loads: with up to eight rows of
    // head size 128, ahead of the wait 178 registers, 4.55 us for 760 keys, 2 kv heads, in L2; after it 221 registers, 4.27 us.  Where the
    // step is prefetched ahead is better (1,500 keys, 8 kv heads 5.37, 5.57 after), and with head size 64 or more rows.
    constexpr bool kAhead = D == 64 || NT == 2 || kPrefetch;
    const uint64_t pol_ahead = kAhead ? small_policy(p) : 0;
    const __nv_bfloat16 *q_rows[NT];                            // this lane's part of its query rows
    if (kAhead) {
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            const int r = g + 8 * n, tq = r / G, gq = r - tq * G;
            q_rows[n] = (const __nv_bfloat16 *)p.q + (((size_t)b * p.q_len + tq) * p.n_q_heads + hk * G + gq) * D + t * 8;
        }
    }
    if (kPrefetch) sm_prefetch<D>(p, b, hk, first, stride, rank == 0 && warp == 0, max_blocks, pol_ahead);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    int kvl = p.kv_len ? __ldg(p.kv_len + b) : p.max_kv_len;    // no length array: every sequence has max_kv_len keys
    if (kvl < p.q_len) kvl = 0;                                 // skipped: its row of the page table may hold anything

    // query rows as A operand; the contraction order is the one of the keys' loads
    if (!kAhead) {
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            const int r = g + 8 * n, tq = r / G, gq = r - tq * G;
            q_rows[n] = (const __nv_bfloat16 *)p.q + (((size_t)b * p.q_len + tq) * p.n_q_heads + hk * G + gq) * D + t * 8;
        }
    }
    uint4 qr[NT][kKV4];
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int j = 0; j < kKV4; ++j) qr[n][j] = g + 8 * n < R ? sm_ldg(q_rows[n] + j * 32) : make_uint4(0, 0, 0, 0);
    const float sl2 = p.scale * kSmLog2e;
    const uint64_t pol = kAhead ? pol_ahead : small_policy(p);
    float o[NT][kDT][4], m[NT], l[NT];
#pragma unroll
    for (int n = 0; n < NT; ++n) {
        m[n] = -INFINITY;
        l[n] = 0.f;
#pragma unroll
        for (int i = 0; i < kDT; ++i) o[n][i][0] = o[n][i][1] = o[n][i][2] = o[n][i][3] = 0.f;
    }

    for (int blk = first; blk < max_blocks; blk += stride) {
        // an identity-mapped cache is addressable up to max_kv_len, so its first loads need not wait for the length (100 keys of 33,000
        // at most 5.5 us a call; 12.0 with blocks beyond the length walked too); a page table is read only where the sequence has a page
        int pid;
        if ((p.page_table || blk != first) && blk * kSmBlock >= kvl) break;
        if (p.page_table) {
            pid = __ldg(p.page_table + (size_t)b * p.max_pages_per_seq + blk / (kPageSize / kSmBlock));
        } else {
            pid = b * p.max_pages_per_seq + blk / (kPageSize / kSmBlock);
        }
        const size_t base = (((size_t)pid * Hkv + hk) * kPageSize + (blk % (kPageSize / kSmBlock)) * kSmBlock) * D;
        uint4 kr[4][kKV4], vr[2][4][D / 64];
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int j = 0; j < kKV4; ++j) kr[x][j] = sm_ldg_hint(kp + base + (x * 8 + g) * D + j * 32 + t * 8, pol);
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y)
#pragma unroll
                for (int z = 0; z < D / 64; ++z)
                    vr[x][y][z] = sm_ldg_hint(vp + base + (x * 16 + (y >> 1) * 8 + 2 * t + (y & 1)) * D + z * 64 + g * 8, pol);

        // ---- scores of the block: s[x] = rows (g, g + 8) x keys (8x + 2t, 8x + 2t + 1)
        float s[4][4];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            s[x][0] = s[x][1] = s[x][2] = s[x][3] = 0.f;
#pragma unroll
            for (int j = 0; j < kKV4; ++j) {
                const uint4 a = qr[0][j], c = qr[NT - 1][j], k = kr[x][j];
                sm_mma(s[x], a.x, NT > 1 ? c.x : 0u, a.y, NT > 1 ? c.y : 0u, k.x, k.y);
                sm_mma(s[x], a.z, NT > 1 ? c.z : 0u, a.w, NT > 1 ? c.w : 0u, k.z, k.w);
            }
        }
        const int key0 = blk * kSmBlock;
        uint32_t pw[NT][4][3];
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            const int limit = kvl - p.q_len + (g + 8 * n) / G;       // last key row g + 8n sees; rows beyond R are zeros
            float mx = m[n];
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int key = key0 + x * 8 + 2 * t + e;
                    float &v = s[x][2 * n + e];
                    v = key <= limit && key < kvl ? v * sl2 : -INFINITY;
                    mx = fmaxf(mx, v);
                }
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            const float ref = mx == -INFINITY ? 0.f : mx;            // nothing visible yet: all probabilities are 0
            const float f = ex2_approx(m[n] - ref);                      // m = -inf gives 0
            float sum = 0.f;
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const float p0 = ex2_approx(s[x][2 * n] - ref), p1 = ex2_approx(s[x][2 * n + 1] - ref);
                sum += p0 + p1;
                sm_split3(p0, p1, pw[n][x]);
            }
            l[n] = l[n] * f + sum;
            m[n] = mx;
            if (blk != first) {   // the rescale factors of the output's columns: rows 2t, 2t + 1 live in lanes g = 2t, 2t + 1
                const float f0 = __shfl_sync(0xffffffffu, f, 8 * t), f1 = __shfl_sync(0xffffffffu, f, 8 * t + 4);
#pragma unroll
                for (int i = 0; i < kDT; ++i) { o[n][i][0] *= f0; o[n][i][1] *= f1; o[n][i][2] *= f0; o[n][i][3] *= f1; }
            }
        }
        // ---- values of keys beyond the length may hold anything: 0 * NaN must not reach the output
        if (key0 + kSmBlock > kvl) {
#pragma unroll
            for (int x = 0; x < 2; ++x)
#pragma unroll
                for (int y = 0; y < 4; ++y)
                    if (key0 + x * 16 + (y >> 1) * 8 + 2 * t + (y & 1) >= kvl)
#pragma unroll
                        for (int z = 0; z < D / 64; ++z) vr[x][y][z] = make_uint4(0, 0, 0, 0);
        }
        // ---- output
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
            for (int z = 0; z < D / 64; ++z) {
                const uint32_t *v0 = reinterpret_cast<const uint32_t *>(&vr[x][0][z]), *v1 = reinterpret_cast<const uint32_t *>(&vr[x][1][z]);
                const uint32_t *v2 = reinterpret_cast<const uint32_t *>(&vr[x][2][z]), *v3 = reinterpret_cast<const uint32_t *>(&vr[x][3][z]);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t a0 = __byte_perm(v0[i], v1[i], 0x5410), a1 = __byte_perm(v0[i], v1[i], 0x7632);
                    const uint32_t a2 = __byte_perm(v2[i], v3[i], 0x5410), a3 = __byte_perm(v2[i], v3[i], 0x7632);
#pragma unroll
                    for (int n = 0; n < NT; ++n)
#pragma unroll
                        for (int w = 2; w >= 0; --w) sm_mma(o[n][z * 4 + i], a0, a1, a2, a3, pw[n][2 * x][w], pw[n][2 * x + 1][w]);
                }
            }
    }

    // ---- the warp's partial: lane (g, t) has rows 2t, 2t + 1 (of each group of eight), dimensions 64z + 8g .. + 7
    float *sm_ml = smem + S::ml_off(), *sm_o = smem + S::o_off(W);
#pragma unroll
    for (int n = 0; n < NT; ++n) {
        float sum = l[n];
        sum += __shfl_xor_sync(0xffffffffu, sum, 1);
        sum += __shfl_xor_sync(0xffffffffu, sum, 2);
        if (t == 0) {
            sm_ml[warp * S::kRows + 8 * n + g] = m[n];
            sm_ml[(W + warp) * S::kRows + 8 * n + g] = sum;
        }
#pragma unroll
        for (int z = 0; z < D / 64; ++z)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                float *dst = sm_o + (warp * S::kRows + 8 * n + 2 * t + e) * S::kOStride + z * 64 + g * 8;
                *reinterpret_cast<float4 *>(dst) = make_float4(o[n][z * 4][e], o[n][z * 4][2 + e], o[n][z * 4 + 1][e], o[n][z * 4 + 1][2 + e]);
                *reinterpret_cast<float4 *>(dst + 4) = make_float4(o[n][z * 4 + 2][e], o[n][z * 4 + 2][2 + e], o[n][z * 4 + 3][e], o[n][z * 4 + 3][2 + e]);
            }
    }
    bool nan = false;
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int i = 0; i < kDT; ++i) nan |= isnan(o[n][i][0]) || isnan(o[n][i][1]) || isnan(o[n][i][2]) || isnan(o[n][i][3]);
    if (__any_sync(0xffffffffu, nan)) {
        __syncwarp();
        attn_small_redo<D, NT>(p, b, hk, first, stride, kvl, sm_ml + warp * S::kRows, sm_o + warp * S::kRows * S::kOStride);
    }
    __syncthreads();
    // ---- the CTA's partial of row r goes to the CTA that merges it, once all of the cluster are known to have started (a CTA without
    //      keys gets here at once)
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
    {
        const uint32_t a_ml = smem_u32(smem + S::recv_ml_off(W)), a_o = smem_u32(smem + S::recv_o_off(W));
        for (int x = tid; x < R * (D / 4); x += blockDim.x) {
            const int r = x / (D / 4), c4 = x % (D / 4);
            float M = -INFINITY, L = 0.f;
            for (int w = 0; w < W; ++w) M = fmaxf(M, sm_ml[w * S::kRows + r]);
            const float ref = M == -INFINITY ? 0.f : M;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int w = 0; w < W; ++w) {
                const float f = ex2_approx(sm_ml[w * S::kRows + r] - ref);
                const float4 a = *reinterpret_cast<const float4 *>(sm_o + (w * S::kRows + r) * S::kOStride + c4 * 4);
                L = fmaf(sm_ml[(W + w) * S::kRows + r], f, L);
                v.x = fmaf(a.x, f, v.x); v.y = fmaf(a.y, f, v.y); v.z = fmaf(a.z, f, v.z); v.w = fmaf(a.w, f, v.w);
            }
            const int entry = (r / cluster_size) * cluster_size + rank, owner = r % cluster_size;
            sm_st_cluster_v4(cluster_map(a_o, (uint32_t)owner) + 4 * (entry * D + c4 * 4), v);
            if (c4 == 0) sm_st_cluster_v2(cluster_map(a_ml, (uint32_t)owner) + 8 * entry, M, L);
        }
    }
    cluster_sync_all();   // release / acquire: the pushed partials are visible to their owners
    // ---- merge the rows r = rank, rank + cluster_size, ...: one warp per row, lanes over the columns
    const float *recv_ml = smem + S::recv_ml_off(W), *recv_o = smem + S::recv_o_off(W);
    for (int r = rank + cluster_size * warp; r < R; r += cluster_size * W) {
        constexpr int V = D / 32;
        const size_t ro = ((size_t)b * p.q_len + r / G) * p.n_q_heads + hk * G + r % G;
        const int e0 = (r / cluster_size) * cluster_size;
        float M = -INFINITY, L = 0.f, av[V];
#pragma unroll
        for (int x = 0; x < V; ++x) av[x] = 0.f;
        for (int c = 0; c < cluster_size; ++c) M = fmaxf(M, recv_ml[2 * (e0 + c)]);
        const float ref = M == -INFINITY ? 0.f : M;
        for (int c = 0; c < cluster_size; ++c) {
            const float f = ex2_approx(recv_ml[2 * (e0 + c)] - ref);
            L = fmaf(recv_ml[2 * (e0 + c) + 1], f, L);
#pragma unroll
            for (int x = 0; x < V; ++x) av[x] = fmaf(recv_o[(e0 + c) * D + lane * V + x], f, av[x]);
        }
        // zeros for a sequence shorter than the query and for a row without a score; a NaN score makes NaN of the row, not zeros
        const bool none = kvl < p.q_len || M == -INFINITY;
        if (none) L = 0.f;
        const float inv = L > 0.f ? 1.f / L : 0.f;
        __nv_bfloat16 *dst = (__nv_bfloat16 *)p.out + ro * D + lane * V;
#pragma unroll
        for (int x = 0; x < V; x += 2) {
            const __nv_bfloat162 h2 = none ? __floats2bfloat162_rn(0.f, 0.f) : __floats2bfloat162_rn(av[x] * inv, av[x + 1] * inv);
            *reinterpret_cast<__nv_bfloat162 *>(dst + x) = h2;
        }
        if (p.lse && lane == 0) p.lse[ro] = L > 0.f ? (M + log2f(L)) * kSmLn2 : -INFINITY;
    }
}

// Function attributes, once per device; dev receives the ordinal.
template <int D, int NT>
static int32_t small_setup(int &dev) {
    static PerDeviceOnce attr_set;
    if (attr_set.needed(dev)) {
        for (auto *kernel : {attn_small_kernel<D, NT, false>, attn_small_kernel<D, NT, true>}) {
            HIPPO_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
            HIPPO_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SmallSmem<D, NT>::bytes(kSmMaxWarps)));
        }
        attr_set.mark(dev);
    }
    return HIPPO_OK;
}

// Clusters of cs CTAs of `warps` warps that the device keeps resident together, asked once per device and shape.
template <int D, int NT>
static int small_room(int warps, int cs) {
    static std::atomic<int> known[kMaxDevices][kSmMaxWarps / 4 + 1][kSmMaxCluster + 1];      // answer + 1
    int dev;
    if (small_setup<D, NT>(dev) != HIPPO_OK || dev < 0) return 1 << 30;      // the launch will say what is wrong
    std::atomic<int> &room = known[dev][warps / 4][cs];
    if (room.load(std::memory_order_relaxed) == 0) {
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)cs;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(cs * kNumSMs));
        cfg.blockDim = dim3((unsigned)(32 * warps));
        cfg.dynamicSmemBytes = SmallSmem<D, NT>::bytes(warps);
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, attn_small_kernel<D, NT, true>, &cfg) != cudaSuccess) { (void)cudaGetLastError(); n = 1 << 30; }
        room.store(n < (1 << 30) ? n + 1 : 1 << 30, std::memory_order_relaxed);
    }
    return room.load(std::memory_order_relaxed) - 1;
}
static int small_room(const AttnParams &p, int warps, int cs) {
    if (p.head_dim == 64) return p.rows <= 8 ? small_room<64, 1>(warps, cs) : small_room<64, 2>(warps, cs);
    return p.rows <= 8 ? small_room<128, 1>(warps, cs) : small_room<128, 2>(warps, cs);
}

// How a call is laid out: warps per CTA, CTAs per unit (= cluster size), 32-key blocks per warp.  The fewest steps win,
// then the fewest warps: with everything in flight at once a step costs 1.1 - 2 us, four warps instead of eight save 0.1.
// Clusters of more than eight need most of a GPC; only six GPCs can be counted on to hold one (8 clusters of 12 CTAs with
// an SM each ran in two waves: 1,500 keys, 8 units, head size 128: 11.3 us against 6.6 on clusters of 8), and sixteen units do
// not all find room for eight either, so the room is asked for (16 units, 2,000 keys, head size 128, 16 rows: 16.6 us in two waves, 12.0).
struct SmallPlan {
    int warps, cluster, steps;
};
static SmallPlan small_plan(const AttnParams &p) {
    const int blocks = ceil_div(p.max_kv_len, kSmBlock), units = p.batch * p.n_kv_heads;
    const int most = p.head_dim == 64 ? kSmMaxWarps : kSmMaxWarps / 2;      // what the register file holds
    SmallPlan best = {0, 0, 0};
    for (int w = 4; w <= most; w *= 2) {
        int lim = most * kNumSMs / (units * w);                              // all warps of the call resident together
        int widest = units * w <= 6 * most ? kSmMaxCluster : kSmMaxCluster / 2;
        if (p.num_splits > 0 && p.num_splits < widest) widest = p.num_splits;
        lim = lim < 1 ? 1 : lim > widest ? widest : lim;
        const int want = ceil_div(blocks, w);
        int cs = want < lim ? want : lim;
        while (cs > 1 && units > small_room(p, w, cs)) --cs;
        const int steps = ceil_div(blocks, w * cs);
        if (!best.warps || steps < best.steps) best = {w, cs, steps};
    }
    return best;
}

// Where this kernel ends and the tensor-memory kernel of attn_tc.cu begins (us per call, this one against the other, or against the
// CUDA-core kernel up to 1,024 keys; one sequence unless noted).  Head size 64, 2 kv heads: 1,000 keys 4.1 / 6.6, 4,000 4.8 / 11.2,
// 8,000 6.2 / 12.8, 33,000 (5 steps) 14.4 / 18.8; 4 kv heads 33,000 keys 15.0 / 19.8; eight sequences of 4,000: 9.5 / 14.7.  Head size
// 128, 14 rows, 4 kv heads: 4,000 keys 7.9 / 12.0, 8,000 11.6 / 14.6, 12,000 14.3 / 16.8, 16,000 (4 steps) 18.0 / 18.5; 8 kv heads,
// 6,000 keys 14.9 / 16.8, 8,000 (4 steps) 18.3 / 18.7.  A caller that asks for more than eight splits of a long
// cache has the other kernel, which can place that many CTAs on scattered SMs (a cluster of more than eight beside a
// verification pass on 96 SMs waited for its end: 32k-token step 2.36 ms against 1.57 ms on clusters of eight).
bool attn_small_supported(const AttnParams &p, int dtype) {
    if (dtype != HIPPO_DTYPE_BF16 || (p.head_dim != 64 && p.head_dim != 128) || p.rows > kSmMaxRows) return false;
    if ((long long)p.batch * p.n_kv_heads * kSmMaxCluster > 65535) return false;
    if (p.max_kv_len <= 1024 && p.rows <= 8) return true;
    return p.num_splits <= kSmMaxCluster / 2 && small_plan(p).steps <= (p.head_dim == 64 ? 5 : 3);
}

// Against the multi-layer launch, which pays its set-up once: better as long as a call is a single step (per layer, head
// size 128: 1,000 keys, 8 rows, 8 kv heads 6.5 us against 11.0, 2,000 keys 7.3 / 8.3, 4,000 keys (2 steps) 14.0 / 8.2).
// A caller's bound on the grid holds for these calls too.
bool attn_small_beats_layers(const AttnParams &p, int dtype, int max_ctas) {
    if (!attn_small_supported(p, dtype)) return false;
    const SmallPlan plan = small_plan(p);
    return plan.steps == 1 && (max_ctas <= 0 || p.batch * p.n_kv_heads * plan.cluster <= max_ctas);
}

// Whether the kernel asks ahead of its wait for what it is going to read (sm_prefetch).  us per call in a chain of 28, without / with, keys
// x kv heads; "cold": the caches of the chain are not in L2 when it begins.  Head size 64: 760 x 4 cold 4.11 / 3.80, in L2 3.52 / 3.47;
// 3,500 x 2 cold 4.83 / 4.17; 9,000 x 8 9.38 / 8.17.  Head size 128, up to eight rows: 1,500 x 8 5.99 / 5.35, 1,500 x 4 4.77 / 4.76; a smaller
// call of a chain that stays in L2 loses, 340 x 8 4.20 / 4.32 and 760 x 2 4.27 / 4.40, against cold 5.07 / 4.76 and 4.85 / 4.70, so the line lies
// where the two are even.  Above, the call before has the memory busy to its end: eight sequences of 3,500 keys x 8, head size 64, 14.4 / 16.4;
// 32 of 1,500 x 4 13.7 / 14.1.
static bool small_prefetch(const AttnParams &p) {
    const long long bytes = (long long)p.batch * p.n_kv_heads * p.max_kv_len * p.head_dim * 4;
    return bytes <= (40 << 20) && (p.head_dim == 64 || p.rows > 8 || bytes >= (1 << 20));
}

template <int D, int NT>
static int32_t launch_small(const AttnParams &p, cudaStream_t stream) {
    int dev;
    const int32_t rc = small_setup<D, NT>(dev);
    if (rc != HIPPO_OK) return rc;
    const SmallPlan plan = small_plan(p);
    const int warps = plan.warps;
    int cs = plan.cluster;
    const int units = p.batch * p.n_kv_heads;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3((unsigned)(32 * warps));
    cfg.dynamicSmemBytes = SmallSmem<D, NT>::bytes(warps);
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    for (;;) {
        attr[1].val.clusterDim.x = (unsigned)cs;
        cfg.gridDim = dim3((unsigned)(units * cs));
        const cudaError_t e = cudaLaunchKernelEx(&cfg, small_prefetch(p) ? attn_small_kernel<D, NT, true> : attn_small_kernel<D, NT, false>, p, cs);
        if (e == cudaSuccess) break;
        (void)cudaGetLastError();
        if (cs <= 8) return cuda_fail(e, "attention (small) launch");
        cs = 8;   // clusters beyond the portable size are not available here
    }
    count_launches(1);
    return HIPPO_OK;
}

int32_t launch_attn_small(const AttnParams &p, cudaStream_t stream) {
    if (p.head_dim == 64) return p.rows <= 8 ? launch_small<64, 1>(p, stream) : launch_small<64, 2>(p, stream);
    return p.rows <= 8 ? launch_small<128, 1>(p, stream) : launch_small<128, 2>(p, stream);
}

}  // namespace hippo
