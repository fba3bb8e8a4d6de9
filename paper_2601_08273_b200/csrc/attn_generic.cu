// CUDA-core split-KV attention (fp32 arithmetic, fp32 or bf16 storage) and the split combine.
//
// Computes softmax(scale * q K^T) V with grouped-query attention and a bottom-right-aligned causal tail
// (Section 3.2: the drafting and verification forward passes attend over the KV cache).  This is the path for
// fp32 caches (the tiny configuration, 1e-5 tolerance) and for shapes the tensor-core kernel does not cover.
//
// Grid (split, kv_head, batch); 8 warps.  A CTA streams tiles of 32 keys of its split, consecutive ones, through shared memory (16 where
// the rows leave no room); packed row r = t*G + g: query token t, head g of the group.  Per tile: a thread per (row, key) forms a score,
// a warp per row updates the row's maximum and sum, a thread per (row, four columns) updates the output (online softmax).
// Up to 16 splits form a cluster and merge through distributed shared memory, which takes one launch; more (long caches, few
// units) go through partial slots and the combine kernel.  Bound: latency at the sizes it serves (the tiny configuration: 62
// keys 4 us a call, 18 us with a serial dot product per lane, rows in turn and always the second kernel).
#include <math.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace hippo {

constexpr int kGenThreads = 256;
constexpr int kGenWarps = kGenThreads / 32;
constexpr int kGenMaxCluster = 16;

__device__ __forceinline__ float4 load_kv4(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }
__device__ __forceinline__ float4 load_kv4(const __nv_bfloat16 *p) {
    const uint2 u = __ldg(reinterpret_cast<const uint2 *>(p));
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.x)), b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&u.y));
    return make_float4(a.x, a.y, b.x, b.y);
}

// Shared memory of a CTA, in floats: Q[R][D] | O[R][D] | K[tile][D + 4] | V[tile][D + 4] | P[R][tile] | m[R] | l[R] | rescale[R]
__host__ __device__ inline size_t generic_smem_floats(int R, int D, int tile) {
    return 2 * (size_t)R * D + 2 * (size_t)tile * (D + 4) + (size_t)R * tile + 3 * (size_t)R;
}

// kEarly: identity-mapped cache, a tile per CTA at most and small enough for kEarlyLoads registers of K and V per thread.  Such a cache is
// addressable up to max_kv_len, so the tile need not wait for the length.  The whole step on the tiny configuration, 4 heads, 290 keys:
// 49.2 us without, 46.4 with.  A kernel of its own: in the general one the held tile cost every other shape 3-17 %.
constexpr int kEarlyLoads = 2;
template <typename T, bool kEarly>
__global__ void __launch_bounds__(kGenThreads) attn_generic_kernel(const AttnParams p, const int tile_keys, const int cluster) {
    extern __shared__ __align__(16) float smem[];
    const int D = p.head_dim, R = p.rows, G = p.group, KS = D + 4;
    float *Qs = smem, *Os = Qs + (size_t)R * D, *Ks = Os + (size_t)R * D, *Vs = Ks + tile_keys * KS, *Ps = Vs + tile_keys * KS;
    float *ms = Ps + (size_t)R * tile_keys, *ls = ms + R, *fs = ls + R;
    const int split = blockIdx.x, hk = blockIdx.y, b = blockIdx.z;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const T *kp = (const T *)p.k_pages, *vp = (const T *)p.v_pages;
    const int D4 = D / 4;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    float4 k_early[kEarlyLoads], v_early[kEarlyLoads];
    if (kEarly && split * tile_keys < p.max_kv_len) {
        const int tok0 = split * tile_keys;
        const size_t base = (((size_t)(b * p.max_pages_per_seq + tok0 / kPageSize) * p.n_kv_heads + hk) * kPageSize + tok0 % kPageSize) * D;
#pragma unroll
        for (int e = 0; e < kEarlyLoads; ++e) {
            const int i = tid + e * kGenThreads;
            if (i < tile_keys * D4) { k_early[e] = load_kv4(kp + base + (size_t)i * 4); v_early[e] = load_kv4(vp + base + (size_t)i * 4); }
        }
    }
    const int kvl = p.kv_len ? p.kv_len[b] : p.max_kv_len;
    const bool skipped = kvl < p.q_len;                     // zeros; the combine kernel writes them where there is one
    if (skipped && !cluster) return;

    const T *q = (const T *)p.q;
    for (int i = tid; i < R * D; i += kGenThreads) {
        const int r = i / D, d = i % D, t = r / G, g = r % G;
        Qs[i] = to_float(q[(((size_t)b * p.q_len + t) * p.n_q_heads + hk * G + g) * D + d]);
        Os[i] = 0.f;
    }
    for (int r = tid; r < R; r += kGenThreads) { ms[r] = -INFINITY; ls[r] = 0.f; }

    const int n_splits = cluster ? cluster : p.num_splits;
    const int n_tiles = skipped ? 0 : (kvl + tile_keys - 1) / tile_keys;
    const int per = kEarly ? 1 : (n_tiles + n_splits - 1) / n_splits;
    const int t0 = split * per, t1 = min(n_tiles, t0 + per);

    for (int tile = t0; tile < t1; ++tile) {
        const int tok0 = tile * tile_keys;
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        if (kEarly) {
#pragma unroll
            for (int e = 0; e < kEarlyLoads; ++e) {
                const int i = tid + e * kGenThreads, j = i / D4, d = (i % D4) * 4;
                if (i >= tile_keys * D4) continue;
                const bool ok = tok0 + j < kvl;
                *reinterpret_cast<float4 *>(Ks + j * KS + d) = ok ? k_early[e] : z;
                *reinterpret_cast<float4 *>(Vs + j * KS + d) = ok ? v_early[e] : z;
            }
        } else {
            const int pid = page_of(p.page_table, p.max_pages_per_seq, b, tok0 / kPageSize);
            const size_t base = (((size_t)pid * p.n_kv_heads + hk) * kPageSize + (tok0 % kPageSize)) * D;
            for (int i = tid; i < tile_keys * D4; i += kGenThreads) {
                const int j = i / D4, d = (i % D4) * 4;
                const bool ok = tok0 + j < kvl;
                const float4 k = ok ? load_kv4(kp + base + (size_t)j * D + d) : z, v = ok ? load_kv4(vp + base + (size_t)j * D + d) : z;
                *reinterpret_cast<float4 *>(Ks + j * KS + d) = k;
                *reinterpret_cast<float4 *>(Vs + j * KS + d) = v;
            }
        }
        __syncthreads();
        // ---- scores
        for (int i = tid; i < R * tile_keys; i += kGenThreads) {
            const int r = i / tile_keys, j = i % tile_keys;
            const int limit = kvl - p.q_len + r / G;        // last visible key of this row
            float s = -INFINITY;
            if (tok0 + j <= limit) {
                float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
                const float4 *qr = reinterpret_cast<const float4 *>(Qs + (size_t)r * D), *kr = reinterpret_cast<const float4 *>(Ks + j * KS);
#pragma unroll 8
                for (int d = 0; d < D4; ++d) {
                    const float4 x = qr[d], y = kr[d];
                    a.x = fmaf(x.x, y.x, a.x); a.y = fmaf(x.y, y.y, a.y); a.z = fmaf(x.z, y.z, a.z); a.w = fmaf(x.w, y.w, a.w);
                }
                s = ((a.x + a.y) + (a.z + a.w)) * p.scale;
            }
            Ps[i] = s;
        }
        __syncthreads();
        // ---- running maxima and sums
        for (int r = warp; r < R; r += kGenWarps) {
            const float s = lane < tile_keys ? Ps[r * tile_keys + lane] : -INFINITY;
            float tmax = s;
#pragma unroll
            for (int o = 16; o; o >>= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
            const float m_old = ms[r], m_new = fmaxf(m_old, tmax);
            const float pj = (s == -INFINITY) ? 0.f : expf(s - m_new);                 // nothing visible yet: all zeros
            const float corr = (m_old == -INFINITY) ? 0.f : expf(m_old - m_new);
            float psum = pj;
#pragma unroll
            for (int o = 16; o; o >>= 1) psum += __shfl_xor_sync(0xffffffffu, psum, o);
            if (lane < tile_keys) Ps[r * tile_keys + lane] = pj;
            __syncwarp();
            if (lane == 0) { ms[r] = m_new; ls[r] = ls[r] * corr + psum; fs[r] = corr; }
        }
        __syncthreads();
        // ---- output
        for (int i = tid; i < R * D4; i += kGenThreads) {
            const int r = i / D4, d = (i % D4) * 4;
            float4 *op = reinterpret_cast<float4 *>(Os + (size_t)r * D + d);
            const float f = fs[r];
            float4 a = *op;
            a.x *= f; a.y *= f; a.z *= f; a.w *= f;
            const float *pr = Ps + r * tile_keys;
#pragma unroll 8
            for (int j = 0; j < tile_keys; ++j) {
                const float4 v = *reinterpret_cast<const float4 *>(Vs + j * KS + d);
                const float w = pr[j];
                a.x = fmaf(w, v.x, a.x); a.y = fmaf(w, v.y, a.y); a.z = fmaf(w, v.z, a.z); a.w = fmaf(w, v.w, a.w);
            }
            *op = a;
        }
        __syncthreads();
    }
    if (!cluster) {
        __syncthreads();
        float *slot = p.partials + ((size_t)(b * p.n_kv_heads + hk) * p.num_splits + split) * slot_float_count(R, D);
        const int Rp = slot_rows_padded(R);
        for (int r = tid; r < R; r += kGenThreads) { slot[r] = ms[r]; slot[Rp + r] = ls[r]; }
        for (int i = tid; i < R * D; i += kGenThreads) slot[2 * Rp + i] = Os[i];
        return;
    }
    // ---- merge: row r by CTA r mod cluster, a warp per row; lane c reads CTA c's maximum and sum
    cluster_sync_all();
    for (int r = split + cluster * warp; r < R; r += cluster * kGenWarps) {
        const uint32_t peer = (uint32_t)(lane < cluster ? lane : 0);
        const float m = lane < cluster ? ld_cluster_f32(cluster_map(smem_u32(ms + r), peer)) : -INFINITY;
        const float l = lane < cluster ? ld_cluster_f32(cluster_map(smem_u32(ls + r), peer)) : 0.f;
        float M = m;
#pragma unroll
        for (int o = 16; o; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
        const float f = m == -INFINITY ? 0.f : expf(m - M);
        float L = l * f;
#pragma unroll
        for (int o = 16; o; o >>= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
        if (skipped) L = 0.f;
        const float inv = L > 0.f ? 1.f / L : 0.f;
        const size_t row = ((size_t)b * p.q_len + r / G) * p.n_q_heads + hk * G + r % G;
        for (int d = lane; d < D; d += 32) {
            float x[kGenMaxCluster], acc = 0.f;
#pragma unroll
            for (int c = 0; c < kGenMaxCluster; ++c) x[c] = c < cluster ? ld_cluster_f32(cluster_map(smem_u32(Os + (size_t)r * D + d), (uint32_t)c)) : 0.f;
#pragma unroll
            for (int c = 0; c < kGenMaxCluster; ++c) {
                const float fc = __shfl_sync(0xffffffffu, f, c);
                if (fc != 0.f) acc = fmaf(x[c], fc, acc);
            }
            store_from_float((T *)p.out + row * D + d, skipped ? 0.f : acc * inv);
        }
        if (p.lse && lane == 0) p.lse[row] = L > 0.f ? M + logf(L) : -INFINITY;
    }
    cluster_sync_all();                                     // nobody leaves while its shared memory is read
}

// One warp per output row (b, t, h): merge the per-split (m, l, O) partials of its (b, kv head).
// Slots of one (b, kv head) are the n_splits consecutive slots starting at (b*H_kv + hk) * n_splits.
template <typename T>
__global__ void attn_combine_kernel(const AttnParams p, int n_splits) {
    const int D = p.head_dim, R = p.rows, G = p.group;
    const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const int total = p.batch * p.q_len * p.n_q_heads;
    if (row >= total) return;
    const int h = row % p.n_q_heads, t = (row / p.n_q_heads) % p.q_len, b = row / (p.n_q_heads * p.q_len);
    const int hk = h / G, r = t * G + (h % G);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    T *out = (T *)p.out + (size_t)row * D;
    if ((p.kv_len ? p.kv_len[b] : p.max_kv_len) < p.q_len) {
        for (int d = lane; d < D; d += 32) store_from_float(out + d, 0.f);
        if (p.lse && lane == 0) p.lse[row] = -INFINITY;
        return;
    }
    const size_t slot_floats = slot_float_count(R, D);
    const int Rp = slot_rows_padded(R);
    const float *base = p.partials + (size_t)(b * p.n_kv_heads + hk) * n_splits * slot_floats;
    float M = -INFINITY;
    for (int s = 0; s < n_splits; ++s) M = fmaxf(M, base[s * slot_floats + r]);
    float L = 0.f;
    for (int s = 0; s < n_splits; ++s) {
        float m = base[s * slot_floats + r];
        if (m != -INFINITY) L += base[s * slot_floats + Rp + r] * expf(m - M);
    }
    const float inv = L > 0.f ? 1.f / L : 0.f;
    for (int d = lane; d < D; d += 32) {
        float acc = 0.f;
        for (int s = 0; s < n_splits; ++s) {
            float m = base[s * slot_floats + r];
            if (m != -INFINITY) acc = fmaf(base[s * slot_floats + 2 * Rp + (size_t)r * D + d], expf(m - M), acc);
        }
        store_from_float(out + d, acc * inv);
    }
    if (p.lse && lane == 0) p.lse[row] = M + logf(L);
}

template <typename T, bool kEarly>
static int32_t launch_generic(const AttnParams &p, int tile, int cluster, size_t smem, cudaStream_t stream) {
    static PerDeviceOnce attr_set;
    int dev;
    if (attr_set.needed(dev)) {
        HIPPO_CUDA_TRY(cudaFuncSetAttribute(attn_generic_kernel<T, kEarly>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        HIPPO_CUDA_TRY(cudaFuncSetAttribute(attn_generic_kernel<T, kEarly>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        attr_set.mark(dev);
    }
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kGenThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = cluster ? 2 : 1;
    for (;;) {
        attr[1].val.clusterDim.x = (unsigned)cluster;
        cfg.gridDim = dim3((unsigned)(cluster ? cluster : p.num_splits), (unsigned)p.n_kv_heads, (unsigned)p.batch);
        const cudaError_t e = cudaLaunchKernelEx(&cfg, attn_generic_kernel<T, kEarly>, p, tile, cluster);
        if (e == cudaSuccess) break;
        (void)cudaGetLastError();
        if (cluster <= 8) return cuda_fail(e, "attention (generic) launch");
        // clusters beyond the portable size are not available here
        if (kEarly) return launch_generic<T, false>(p, tile, 8, smem, stream);      // perhaps more than a tile per CTA
        cluster = 8;
    }
    count_launches(1);
    return HIPPO_OK;
}

int32_t launch_attn_generic(const AttnParams &p, int dtype, cudaStream_t stream) {
    int tile = 32;
    size_t smem = generic_smem_floats(p.rows, p.head_dim, tile) * sizeof(float);
    if (smem > 227 * 1024) smem = generic_smem_floats(p.rows, p.head_dim, tile = 16) * sizeof(float);
    if (smem > 227 * 1024) return fail(HIPPO_ERR_UNSUPPORTED_SHAPE, "attention: rows*head_dim too large for shared memory");
    // one launch where a cluster covers the splits, or where it leaves a CTA at most two tiles
    const int cluster = p.num_splits <= kGenMaxCluster ? p.num_splits : ceil_div(p.max_kv_len, tile) <= 2 * kGenMaxCluster ? kGenMaxCluster : 0;
    const bool early = !p.page_table && ceil_div(p.max_kv_len, tile) <= (cluster ? cluster : p.num_splits) && tile * p.head_dim / 4 <= kEarlyLoads * kGenThreads;
    const int32_t rc = dtype == HIPPO_DTYPE_FP32
        ? (early ? launch_generic<float, true>(p, tile, cluster, smem, stream) : launch_generic<float, false>(p, tile, cluster, smem, stream))
        : (early ? launch_generic<__nv_bfloat16, true>(p, tile, cluster, smem, stream) : launch_generic<__nv_bfloat16, false>(p, tile, cluster, smem, stream));
    if (rc != HIPPO_OK || cluster) return rc;
    return launch_attn_combine(p, dtype, p.num_splits, stream);
}

int32_t launch_attn_combine(const AttnParams &p, int dtype, int n_splits, cudaStream_t stream) {
    const int total = p.batch * p.q_len * p.n_q_heads;
    const int warps_per_block = 4;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((total + warps_per_block - 1) / warps_per_block));
    cfg.blockDim = dim3(warps_per_block * 32);
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (dtype == HIPPO_DTYPE_FP32)
        HIPPO_CUDA_TRY(cudaLaunchKernelEx(&cfg, attn_combine_kernel<float>, p, n_splits));
    else
        HIPPO_CUDA_TRY(cudaLaunchKernelEx(&cfg, attn_combine_kernel<__nv_bfloat16>, p, n_splits));
    count_launches(1);
    HIPPO_CUDA_TRY(cudaGetLastError());
    return HIPPO_OK;
}

}  // namespace hippo
