// Norms, temporal dot products and spatial scores of bf16 embeddings (Section 5.1, Eq. 3-6) on the tensor cores, with the
// accuracy of fp64.
//
// The standardisation of the spatial score divides by a sigma of ~1e-4, so Gram entries must be good to ~1e-11 relative to the
// norms; the fp64 tensor instruction gives that at 64 multiply-adds per clock and SM and was the bound of the selection.  Here a
// token's elements are written as
//     x = s (q + r),   s = 2^e per token,  q = 256 H + M an integer of |q| < 2^15 with signed 8-bit digits,  |r| <= 1/2,
// so that   <x_i, x_j> / (s_i s_j) = 65536 <H,H> + 256 (<H_i,M_j> + <M_i,H_j>) + <M,M>      int8 x int8 -> int32, exact
//                                   + C_ij + C_ji,   2 C_ij = sum_k r_i (2 x_j / s_j - r_j)      fp16 x fp16 -> fp32.
// r has at most the 8 significant bits of x and 2 x / s - r nine, so fp16 holds both exactly (bf16 would round the second, by
// an amount that depends on r: 1e-9 of the norms on nearly equal tokens).  The fp32 rounding of C is the only inexact step.  r is
// non-zero only for elements below 2^-8 of the upper bound 2^15 s, 1 in 60 of normal ones, and C is then 2^-20 of the norms or less.
// s must follow the bulk of a token's elements: one large dimension that set it would push the others into r.  It comes from the
// maxima of 16 pieces of 8 elements spread over the token: the bound is 4 - 8 times one of the upper ones (three large dimensions
// among the samples do not move it), but not more than four times as far above one of the lower half, should there be more of them.
// An element above it (a heavy tail, an outlier dimension, infinity or NaN) is taken out (q = r = 0), noted in a list, and its
// products are added in fp64 from memory; a tile with many of them has its sums formed in fp64 throughout.
//
// A tile of 128 rows holds the same crop in floor(128 / crop) consecutive frames, row = frame * crop + cell.  Its 128 x 128
// product contains, besides the crops' Gram matrices on the diagonal, the dot products with the same cell of the next frame on
// the m-th off-diagonal: the temporal score costs no extra pass.  Neighbouring tiles share one frame.
//
// CTA: 16 warps read global memory straight into registers (four steps ahead), split it into the four operands and store them
// in the 128-byte-swizzled layout; a seventeenth issues the MMAs (per 64 dimensions: 2 x [H x (H;M) N = 256, M x M N = 128] in
// kind::i8, 4 x [r x (2x - r)] in kind::f16, 640 clocks).  Four accumulators of 128 columns fill tensor memory.  The CTAs of a
// cluster split the embedding dimension and add their blocks through distributed shared memory.
// Bound: the shared-memory and L1 data path (per step of 64 dimensions 64 KB loaded, stored and passed through L1, 72 KB read by
// the MMAs, 1,270 clocks of the 1,700 that a step takes) beside the conversion (about 150 instructions per thread and step, 940
// clocks with neither loads nor MMAs).  65,536 tokens of 8,192: 440 us; 890 us for the fp64 kernels.  Measured and not better: MMA
// issue by one of the converting warps (+25 %), L2 prefetch ahead of the loads (+6 %), generic instead of shared stores (+10 %).
#include <cuda_fp16.h>
#include <math.h>

#include <type_traits>

#include "select.cuh"
#include "tc_ptx.cuh"

namespace hippo {

constexpr int kGramRows = 128;
constexpr int kGramProducers = 512;
constexpr int kGramThreads = kGramProducers + 32;
constexpr int kGramStep = 64;                    // dimensions per step
constexpr int kGramSlots = 4;                    // steps in the ring of operands
constexpr int kGramAhead = 4;                    // steps that the loads run ahead
constexpr int kGramRTile = kGramRows * 128;      // bytes of a 128-row tile of 128-byte rows
constexpr int kGramList = 6144;                  // elements above the bound that a CTA can note
constexpr int kGramPStride = kMaxCrop + 1;
constexpr int kGramUnit = 127 + 15;              // log2(1 / s) + E
constexpr unsigned long long kGramWaitLimitNs = 2000000000ull;

// A class of equal crops: all inner ones, the clipped ones at the right edge, at the bottom edge, in the corner.
struct GramClass {
    int h, w, n_y, n_x, y0, x0;      // crop size, crops of the class, first cell
    int frames;                      // frames per tile
};
struct GramParams {
    GramClass cls[4];
    int splits;                      // cluster size: CTAs that share a tile's embedding dimensions
    int tile0;                       // first tile of this launch
    int part;                        // 0: the only launch; 1: the full waves, 2: the rest, which starts as SMs fall free
    WsHeader *header;
    int tile_off[kSelMaxBatch + 1];  // first tile of each sequence
};

__host__ __device__ inline int gram_class_tiles(int n_frames, int frames) {     // tiles per crop: neighbours share a frame
    return n_frames <= frames ? 1 : 1 + (n_frames - frames + frames - 2) / (frames - 1);
}

struct GramShared {
    unsigned long long full[kGramSlots], empty[kGramSlots], done;
    uint32_t tmem_base;
    volatile int abort;
    long long limit_ns;              // of the MMA issuer's waits; 0: the built-in limit
    int n_list, fp64;                // large elements noted; 1: the sums are formed in fp64
    int scale_exp[kGramRows];        // biased exponent E of the bound 2^(E - 127) on the elements; s = 2^(E - 127 - 15)
    int token[kGramRows];            // the rows' tokens (-1: none) and first rows of their crops
    int first[kGramRows];
    double inv_root[kGramRows];      // 1 / root of the scaled norm; -1: the norm is not above 0
    uint32_t list[kGramList];        // gram_entry(row, dimension)
};
// The list of large elements.  Entries order by the warp that adds them up, then by dimension, then by row.
constexpr int kGramOwners = 16, kGramOwned = kGramRows / kGramOwners;   // warps that own rows, rows of each
constexpr int kGramColumn = 96;                                         // a dimension of the rows that a warp looks at: 2 kMaxCrop + 8 at most

constexpr size_t kGramRingBytes = (size_t)kGramSlots * 2 * kGramRTile + 2 * 2 * kGramRTile;
constexpr size_t kGramSmemBytes = 1024 + kGramRingBytes + sizeof(GramShared);
// after the loop the ring holds the CTA's block of sums: P[128][33] | next[128] | previous[128]
constexpr size_t kGramScratch = 40 * 1024;       // offset of the memory behind them
static_assert((kGramRows * kGramPStride + 2 * kGramRows) * sizeof(double) <= kGramScratch, "sums end before the scratch memory");
static_assert(kGramScratch + (2 * kGramList + 2 * kGramOwners + 1 + kGramOwners * kGramColumn) * sizeof(uint32_t) <= kGramRingBytes, "two lists fit behind the sums");
static_assert(kGramSmemBytes <= 227 * 1024, "shared memory of an SM");

// Records that a wait gave up.  The header of a selection workspace need not have been zeroed: whatever the status word holds, it is
// overwritten.
__device__ __forceinline__ void gram_give_up(GramShared *sh, WsHeader *hdr, int site) {
    sh->abort = 1;
    if (atomicExch(&hdr->status, (int)HIPPO_ERR_TIMEOUT) != (int)HIPPO_ERR_TIMEOUT) hdr->where = 200 + site;
}

// Bounded wait.  A drain wait guards the exit of the CTA (tensor-core work in flight): it does not give up because another
// wait did.
// Inlined throughout: a call in the loop would move the loads in flight out of their registers.
__device__ __forceinline__ bool gram_wait(GramShared *sh, WsHeader *hdr, unsigned long long *bar, uint32_t parity, int site,
                                          bool draining = false) {
    const uint32_t b = smem_u32(bar);
    if (mbar_try_wait(b, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (uint32_t i = 1;; ++i) {
        if (mbar_try_wait(b, parity)) return true;
        if ((i & 31) == 0) {
            if (!draining && sh->abort) return false;
            if (global_ns() - t0 > kGramWaitLimitNs) {
                gram_give_up(sh, hdr, site);
                return false;
            }
        }
    }
}

// The issuer's wait for operands honours a limit set in the header, which a healthy kernel can be made to run out of: it then polls
// without suspending and looks at the clock every time.
__device__ __forceinline__ bool gram_wait_limited(GramShared *sh, WsHeader *hdr, unsigned long long *bar, uint32_t parity, int site) {
    if (sh->limit_ns <= 0) return gram_wait(sh, hdr, bar, parity, site);
    const unsigned long long t0 = global_ns();
    while (!mbar_test_wait(smem_u32(bar), parity)) {
        if (sh->abort) return false;
        if (global_ns() - t0 > (unsigned long long)sh->limit_ns) { gram_give_up(sh, hdr, site); return false; }
    }
    return true;
}

__device__ __forceinline__ void tc_mma_i8(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// instruction descriptors: signed 8-bit x signed 8-bit -> int32, fp16 x fp16 -> fp32; both operands K-major
__device__ __forceinline__ uint32_t instr_desc_s8(int m, int n) {
    return (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
__device__ __forceinline__ uint32_t instr_desc_f16(int m, int n) { return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24); }

__device__ __forceinline__ void st_shared_v2(uint32_t addr, const uint2 &v) {
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(v.x), "r"(v.y) : "memory");
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, const uint4 &v) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// pairs of floats
__device__ __forceinline__ uint64_t f2_pack(uint32_t lo, uint32_t hi) { return (uint64_t)lo | ((uint64_t)hi << 32); }
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint32_t f2_half(uint64_t a) {
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(__uint_as_float((uint32_t)(a >> 32))), "f"(__uint_as_float((uint32_t)a)));
    return r;
}

// Eight elements of a token -> digits H, M (8 bytes each), r and x' = 2 x / s - r (eight fp16 each).  The conversion is bound by
// the integer pipe (unpacking, byte permutes, packing), so the check for elements above the bound is a sum of q^2 on the FMA
// pipe: one such element makes it 32,640^2 or more (or NaN), eight of the usual size stay far below.
struct GramSplit {
    uint2 h, m;
    uint4 r, x;
    bool large;
};
__device__ __forceinline__ GramSplit gram_split(const uint4 &u, uint64_t inv2) {
    // 1.5 * 2^23 rounds to an integer that sits in the low bits; + 128 turns the low byte into M + 128 and the next into H
    const uint64_t magic2 = f2_pack(0x4B400080u, 0x4B400080u), neg1 = f2_pack(0xBF800000u, 0xBF800000u), neg2 = f2_pack(0xC0000000u, 0xC0000000u);
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
    uint32_t q[4], r[4], x[4];
    uint64_t sq = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint64_t v = f2_pack(w[i] << 16, w[i] & 0xffff0000u);
        const uint64_t t = f2_fma(v, inv2, magic2);
        const uint64_t nq = f2_fma(t, neg1, magic2);                       // -q
        const uint64_t rr = f2_fma(v, inv2, nq);
        sq = f2_fma(nq, nq, sq);
        r[i] = f2_half(rr);
        x[i] = f2_half(f2_fma(nq, neg2, rr));                              // r + 2 q
        q[i] = __byte_perm((uint32_t)t, (uint32_t)(t >> 32), 0x5140);      // M0 M1 H0 H1
    }
    GramSplit o;
    o.m = make_uint2(__byte_perm(q[0], q[1], 0x5410) ^ 0x80808080u, __byte_perm(q[2], q[3], 0x5410) ^ 0x80808080u);
    o.h = make_uint2(__byte_perm(q[0], q[1], 0x7632), __byte_perm(q[2], q[3], 0x7632));
    o.r = make_uint4(r[0], r[1], r[2], r[3]);
    o.x = make_uint4(x[0], x[1], x[2], x[3]);
    o.large = !(__uint_as_float((uint32_t)sq) + __uint_as_float((uint32_t)(sq >> 32)) < 1.0653e9f);
    return o;
}

// The integer whose bits x holds, exactly: 2^52 + 2^31 + i as a bit pattern, minus the constant (the conversion instruction
// runs at a fraction of the rate of the fp64 adds).
__device__ __forceinline__ double int_to_double(float x) {
    return __hiloint2double(0x43300000, __float_as_int(x) ^ (int)0x80000000) - 4503601774854144.0;
}

// Largest magnitude (bf16 bits) that the digits hold: 254/256 of the bound 2^(E - 127).  255/256 would be q = 32,640, whose upper
// digit is 128.
__device__ __forceinline__ uint32_t gram_limit(int scale_exp) { return ((uint32_t)scale_exp << 7) - 2; }

// An entry of the list of large elements.
__device__ __forceinline__ uint32_t gram_entry(int row, int k) { return (uint32_t)(row / kGramOwned) << 19 | (uint32_t)k << 3 | (uint32_t)(row % kGramOwned); }

// Notes the elements of a piece (row r, dimensions k ..) that are above the row's bound and returns the piece without them.  A tile
// that has noted too many goes to fp64: the rest may stay as it is.
__device__ __noinline__ uint4 gram_take_out(GramShared *sh, uint4 u, int r, int k) {
    if (*(volatile int *)&sh->n_list > kGramList) return u;
    const uint32_t limit = gram_limit(sh->scale_exp[r]);
    uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const uint32_t at16 = (e & 1) * 16, mag = (w[e >> 1] >> at16) & 0x7fffu;
        if (mag > limit) {
            const int at = atomicAdd(&sh->n_list, 1);
            if (at < kGramList) sh->list[at] = gram_entry(r, k + e);
            w[e >> 1] &= ~(0xffffu << at16);
        }
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// 2^e as a double, for the exponents that scales and their products of two have
__device__ __forceinline__ double gram_pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }

// Adds the products of the noted elements to the block of sums P[128][33] | next[128] | previous[128].  The entries are sorted first:
// a row's products are then added in the order of their dimensions, whichever thread noted its piece first, and a warp takes a
// dimension of its eight rows together, with the partners' elements fetched once and the sums in registers.  Selection of 32,768 tokens
// of 4,096 with one / 8 / 12 / 30 large dimensions: 227 / 278 / 301 / 422 us (none: 197; with every warp walking the whole list for
// each of its rows 391 / 1,294 / 1,744 us; fp64 kernels 332 throughout).  Called by all threads; false, and nothing added, with more
// than `most` dimensions to fetch.
__device__ __noinline__ bool gram_add_list(GramShared *sh, uint8_t *scratch, double *P, const __nv_bfloat16 *E, int d, int m, int n, int most) {
    static_assert(kGramOwned == 8 && 2 * kMaxCrop + kGramOwned <= kGramColumn, "three bits of an entry; rows of a column");
    uint32_t *bucket = reinterpret_cast<uint32_t *>(scratch), *sorted = bucket + kGramList;
    int *start = reinterpret_cast<int *>(sorted + kGramList), *fill = start + kGramOwners + 1;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid <= kGramOwners) start[tid] = 0;
    __syncthreads();
    for (int e = tid; e < n; e += kGramThreads) atomicAdd(&start[(sh->list[e] >> 19) + 1], 1);
    __syncthreads();
    if (warp == 0) {                                                 // counts -> first entries
        const int c = lane < kGramOwners ? start[lane + 1] : 0;
        int at = c;
        for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, at, o); if (lane >= o) at += v; }
        if (lane < kGramOwners) { fill[lane] = at - c; start[lane + 1] = at; }
    }
    __syncthreads();
    for (int e = tid; e < n; e += kGramThreads) bucket[atomicAdd(&fill[sh->list[e] >> 19], 1)] = sh->list[e];
    __syncthreads();
    for (int e = tid; e < n; e += kGramThreads) {                    // all different: an entry's place is the number of smaller ones
        const uint32_t it = bucket[e];
        int at = start[it >> 19];
        for (int o = start[it >> 19]; o < start[(it >> 19) + 1]; ++o) at += bucket[o] < it ? 1 : 0;
        sorted[at] = it;
    }
    __syncthreads();
    int firsts = 0;                                                  // dimensions to fetch, counted on top of the end of the first bucket
    for (int e = tid; e < n; e += kGramThreads) firsts += e == 0 || sorted[e] >> 3 != sorted[e - 1] >> 3 ? 1 : 0;
    if (firsts) atomicAdd(&fill[0], firsts);
    __syncthreads();
    if (fill[0] - start[1] > most) return false;
    if (warp >= kGramOwners) return true;
    const int e1 = start[warp + 1], r0 = warp * kGramOwned, base = r0 - m;
    float *const col = reinterpret_cast<float *>(fill + kGramOwners) + warp * kGramColumn;
    for (int q0 = 0; q0 < m + 2; q0 += 32) {                         // lanes: a row's crop, then its neighbours in time
        const int q = q0 + lane;
        int at[kGramOwned];                                          // the partner's place in the column, -1: none
        float top[kGramOwned];
        double sum[kGramOwned];
#pragma unroll
        for (int u = 0; u < kGramOwned; ++u) {
            const int r = r0 + u, j = q < m ? sh->first[r] + q : q == m ? r + m : q == m + 1 ? r - m : -1;
            const bool valid = j >= 0 && j < kGramRows && sh->token[j] >= 0 && sh->token[r] >= 0;
            at[u] = valid ? j - base : -1;
            top[u] = valid ? __uint_as_float(gram_limit(sh->scale_exp[j]) << 16) : 0.f;
            sum[u] = 0.0;
        }
        // One dimension at a time: the partners of the warp's rows lie in rows base .. base + 2 m + 7, a lane fetches up to three of them
        // (a single entry's own partners alone); the next dimension's are on their way meanwhile.
        __nv_bfloat16 next[3];
        uint32_t rows = 0;                                           // which of the warp's rows noted the dimension
        auto fetch = [&](int e) {
            const uint32_t it = sorted[min(e + lane, e1 - 1)], k = __shfl_sync(0xffffffffu, it >> 3, 0);
            rows = __reduce_or_sync(0xffffffffu, it >> 3 == k ? 1u << (it & 7u) : 0u);
            const int r = r0 + __ffs(rows) - 1, fr = sh->first[r];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int row = base + 32 * i + lane;
                const bool wanted = row >= 0 && row < kGramRows && 32 * i + lane < 2 * m + kGramOwned &&
                                    ((rows & (rows - 1)) || (row >= fr && row < fr + m) || row == r + m || row == r - m);
                const int tk = wanted ? sh->token[row] : -1;
                next[i] = tk >= 0 ? E[(size_t)tk * d + (k & 0xffffu)] : __ushort_as_bfloat16(0);
            }
        };
        int e = start[warp];
        if (e < e1) fetch(e);
        while (e < e1) {
            __syncwarp();                                            // the column before has been read
#pragma unroll
            for (int i = 0; i < 3; ++i) col[32 * i + lane] = __bfloat162float(next[i]);
            __syncwarp();
            const uint32_t now = rows;
            e += __popc(now);
            if (e < e1) fetch(e);
#pragma unroll
            for (int u = 0; u < kGramOwned; ++u)
                if (now >> u & 1u) {
                    const float x = col[m + u], y = col[max(at[u], 0)];
                    // an element that is in the list for both tokens appears in both orders: half each time
                    sum[u] = fma((double)x, (double)(fabsf(y) <= top[u] ? y : 0.5f * y), sum[u]);
                }
        }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < kGramOwned; ++u)
            if (at[u] >= 0) {
                double *dst = q < m ? P + (r0 + u) * kGramPStride + q : P + kGramRows * kGramPStride + (q == m ? 0 : kGramRows) + r0 + u;
                *dst += sum[u] * gram_pow2(2 * kGramUnit - sh->scale_exp[r0 + u] - sh->scale_exp[base + at[u]]);
            }
    }
    return true;
}

// The block of sums in fp64 throughout, for a tile with more large elements than the list holds (or with tokens below the smallest
// scale): dimensions k0 .. k1 of the rows are staged as doubles, 64 at a time, and warp w multiplies group w of eight rows with the
// groups that its partners (crop and next frame, rows i .. i + m) can lie in, on the fp64 tensor path.  Bound by that instruction:
// 80 of them per four dimensions and tile where crops of 25 need 33.  Selection of 32,768 tokens of 4,096, every tile: 655 us
// (6,500 with a dependent chain per row and partner, 330 with the kernels of select.cu, which share nothing between crops and
// frames but have no tile of 128 rows to fill).  Called by all threads.
constexpr int kGramF64Stride = kGramStep + 4;      // the four rows of a half-warp's fragment load fall into different banks
static_assert(kGramScratch + 2 * kGramRows * kGramF64Stride * sizeof(double) <= kGramRingBytes, "staged rows fit behind the sums");
__device__ __noinline__ void gram_sum_fp64(GramShared *sh, double *stage, double *P, const __nv_bfloat16 *E, int d, int m, int k0, int k1) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, groups = kGramRows / 8;
    const int r = tid >> 2, part = (tid & 3) * 16;                    // staging: a quarter of a row's dimensions per thread
    const int tk = tid < kGramProducers ? sh->token[r] : -1;
    double acc[5][2];
#pragma unroll
    for (int o = 0; o < 5; ++o) acc[o][0] = acc[o][1] = 0.0;
    const int last = (7 + m) / 8;                                     // offset of the last group of partners; m <= 32: 4 at most
    uint4 u[2];
    auto load = [&](int k) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
            u[h] = tk >= 0 && k + part + h * 8 < k1 ? __ldg(reinterpret_cast<const uint4 *>(E + (size_t)tk * d + k + part + h * 8)) : make_uint4(0, 0, 0, 0);
    };
    auto store = [&](int buf) {
        if (tid >= kGramProducers) return;
        double *dst = stage + buf * kGramRows * kGramF64Stride + r * kGramF64Stride + part;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t w[4] = {u[h].x, u[h].y, u[h].z, u[h].w};
#pragma unroll
            for (int i = 0; i < 4; ++i)
                *reinterpret_cast<double2 *>(dst + h * 8 + 2 * i) = make_double2((double)__uint_as_float(w[i] << 16), (double)__uint_as_float(w[i] & 0xffff0000u));
        }
    };
    __syncthreads();
    load(k0);
    store(0);
    load(k0 + kGramStep);
    for (int k = k0, buf = 0; k < k1; k += kGramStep, buf ^= 1) {     // two buffers: a step is stored while the one before is multiplied
        __syncthreads();
        store(buf ^ 1);
        load(k + 2 * kGramStep);
        if (warp < groups) {
            const double *from = stage + buf * kGramRows * kGramF64Stride + (lane >> 2) * kGramF64Stride + (lane & 3);
            // straight-line code per number of groups (a branch per instruction halves the rate); groups past the last row are products
            // of the last one that nobody looks at
            auto multiply = [&](auto count) {
                constexpr int N = decltype(count)::value;
                const double *g[N];
#pragma unroll
                for (int o = 0; o < N; ++o) g[o] = from + min(warp + o, groups - 1) * 8 * kGramF64Stride;
#pragma unroll 4
                for (int s = 0; s < kGramStep; s += 4) {
                    const double x = g[0][s];
#pragma unroll
                    for (int o = 0; o < N; ++o) dmma_m8n8k4(acc[o][0], acc[o][1], x, o ? g[o][s] : x);
                }
            };
            using std::integral_constant;
            if (last >= 4) multiply(integral_constant<int, 5>{});
            else if (last == 3) multiply(integral_constant<int, 4>{});
            else if (last == 2) multiply(integral_constant<int, 3>{});
            else multiply(integral_constant<int, 2>{});
        }
    }
    __syncthreads();
    if (warp < groups) {
        const int i = warp * 8 + (lane >> 2), ti = sh->token[i];
#pragma unroll
        for (int o = 0; o < 5; ++o)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int j = (warp + o) * 8 + (lane & 3) * 2 + e;
                if (o > last || j >= kGramRows || j < i || ti < 0 || sh->token[j] < 0) continue;
                const double v = 0.5 * acc[o][e] * gram_pow2(kGramUnit - sh->scale_exp[i]) * gram_pow2(kGramUnit - sh->scale_exp[j]);
                if (sh->first[i] == sh->first[j]) {
                    P[i * kGramPStride + j - sh->first[j]] = v;
                    P[j * kGramPStride + i - sh->first[i]] = v;
                }
                if (j == i + m) { P[kGramRows * kGramPStride + i] = v; P[kGramRows * (kGramPStride + 1) + j] = v; }
            }
    }
    __syncthreads();
}

// Adds the other CTAs' blocks of sums to rank 0's, in rank order.  All loads of a batch are in flight before the first is used:
// a remote load takes about as long as one from L2.
template <int S, int BATCH>
__device__ __forceinline__ void gram_add_peers(double *P) {
    constexpr int kN = kGramRows * kGramPStride + 2 * kGramRows;
    const uint32_t mine = smem_u32(P);
    for (int i0 = threadIdx.x; i0 < kN; i0 += BATCH * kGramThreads) {
        double w[BATCH][S - 1];
#pragma unroll
        for (int k = 0; k < BATCH; ++k)
#pragma unroll
            for (int q = 1; q < S; ++q) {
                w[k][q - 1] = 0.0;
                if (i0 + k * kGramThreads < kN)
                    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(w[k][q - 1]) : "r"(cluster_map(mine + 8 * (i0 + k * kGramThreads), (uint32_t)q)) : "memory");
            }
#pragma unroll
        for (int k = 0; k < BATCH; ++k) {
            const int i = i0 + k * kGramThreads;
            if (i >= kN) continue;
            double v = P[i];
#pragma unroll
            for (int q = 0; q < S - 1; ++q) v += w[k][q];
            P[i] = v;
        }
    }
}

__global__ void __launch_bounds__(kGramThreads, 1) select_gram_kernel(const SelectParams p, const GramParams gp) {
    extern __shared__ uint8_t gram_smem[];
    uint8_t *ring = (uint8_t *)(((uintptr_t)gram_smem + 1023) & ~(uintptr_t)1023);
    uint8_t *digits = ring + kGramSlots * 2 * kGramRTile;        // [2] H tile | M tile: 128 dimensions, i.e. two steps
    GramShared *sh = (GramShared *)(ring + kGramRingBytes);
    double *P = (double *)ring, *t_next = P + kGramRows * kGramPStride, *t_prev = t_next + kGramRows;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // ---- which tile: sequence, crop class, crop, frames
    const int tile = gp.tile0 + blockIdx.x / gp.splits, rank = blockIdx.x % gp.splits;
    const int b = find_seq(gp.tile_off, p.batch, tile);
    const int n_v = p.seq_off[b + 1] - p.seq_off[b], n_frames = (n_v + p.tpf - 1) / p.tpf;
    int x = tile - gp.tile_off[b], ci = 0, per_crop = 1;
    for (; ci < 3; ++ci) {
        per_crop = gram_class_tiles(n_frames, gp.cls[ci].frames);
        const int n = gp.cls[ci].n_y * gp.cls[ci].n_x * per_crop;
        if (x < n) break;
        x -= n;
    }
    const GramClass c = gp.cls[ci];
    per_crop = gram_class_tiles(n_frames, c.frames);
    const int crop = x / per_crop, f0 = (x % per_crop) * (c.frames - 1);
    const int f1 = min(n_frames, f0 + c.frames);                   // frames [f0, f1) are in the tile
    const int own_end = f1 == n_frames ? f1 : f1 - 1;              // the shared frame belongs to the next tile
    const int y0 = c.y0 + (crop / c.n_x) * p.crop_h, x0 = c.x0 + (crop % c.n_x) * p.crop_w, m = c.h * c.w;
    // token of row r, or -1
    auto token = [&](int r) {
        const int f = f0 + r / m, a = r % m;
        const int cell = (y0 + a / c.w) * p.grid_w + x0 + a % c.w;
        return f < f1 && f * p.tpf + cell < n_v ? p.seq_off[b] + f * p.tpf + cell : -1;
    };
    const __nv_bfloat16 *E = (const __nv_bfloat16 *)p.embeds;

    WsHeader *hdr = gp.header;
    if (token(0) < 0) {                    // a crop beyond the end of a partial frame: nothing here, for any CTA of the cluster
        if (gp.part == 2) asm volatile("griddepcontrol.wait;" ::: "memory");
        return;
    }
    // ---- set-up
    if (tid < kGramSlots) mbar_init(smem_u32(&sh->full[tid]), kGramProducers / 32);
    else if (tid < 2 * kGramSlots) mbar_init(smem_u32(&sh->empty[tid - kGramSlots]), 1);
    else if (tid == 2 * kGramSlots) mbar_init(smem_u32(&sh->done), 1);
    else if (tid == 64) { sh->abort = 0; sh->n_list = 0; sh->fp64 = 0; }
    if (warp == kGramProducers / 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh->tmem_base)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // the second launch begins once every CTA of the first has got here, so what came before both is complete then; it waits for
    // the first at its end, so that whatever follows waits for both
    if (gp.part < 2) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (gp.part == 1) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    bool below = false;           // the row's elements lie below the smallest scale
    int above = 0;                // this thread's pieces with an element above the bound
    if (tid == 512) {             // the header may hold anything: a limit counts only with its key
        const long long limit = hdr->wait_limit_ns;
        sh->limit_ns = hdr->wait_limit_key == (limit ^ kWaitLimitKey) && limit < (long long)kGramWaitLimitNs ? limit : 0;
    }
    if (tid < kGramProducers) {   // the token's scale: 16 pieces of 8 elements spread over it, four per thread
        const int r = tid >> 2, tk = token(r), pieces = p.d / 8;
        uint32_t mx[4] = {0, 0, 0, 0};                               // the pieces' maxima, bf16 bits
        if (tk >= 0) {
            uint4 u[4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
                u[i] = __ldg(reinterpret_cast<const uint4 *>(E + (size_t)tk * p.d) + (long long)pieces * ((tid & 3) * 4 + i) / 16);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t w[4] = {u[i].x, u[i].y, u[i].z, u[i].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t lo = w[e] & 0x7fffu, hi = (w[e] >> 16) & 0x7fffu;
                    if (lo < 0x7f80u) mx[i] = max(mx[i], lo);       // infinities and NaN say nothing about the scale
                    if (hi < 0x7f80u) mx[i] = max(mx[i], hi);
                }
            }
        }
        auto order = [&](int i, int j) { const uint32_t lo = min(mx[i], mx[j]); mx[j] = max(mx[i], mx[j]); mx[i] = lo; };
        order(0, 1); order(2, 3); order(0, 2); order(1, 3); order(1, 2);
        // second largest, second smallest over the row's four threads
        auto second = [&](uint32_t v, bool largest) {
            const uint32_t w = __shfl_xor_sync(0xffffffffu, v, 1), hi = max(v, w), lo = min(v, w);
            const uint32_t hi2 = __shfl_xor_sync(0xffffffffu, hi, 2), lo2 = __shfl_xor_sync(0xffffffffu, lo, 2);
            return largest ? max(min(hi, hi2), max(lo, lo2)) : min(max(lo, lo2), min(hi, hi2));
        };
        // from the upper ones, whatever up to three large dimensions among the samples are; and from the lower half, up to eight
        uint32_t high = second(mx[2], true), mid = second(mx[1], false);
        const uint32_t two = second(mx[3], true);
        uint32_t most = max(mx[3], __shfl_xor_sync(0xffffffffu, mx[3], 1));
        most = max(most, __shfl_xor_sync(0xffffffffu, most, 2));
        if (high == 0) high = two ? two : most;                      // few pieces hold anything but zeros
        if (mid == 0) mid = high;
        // nothing but zeros among the samples says nothing about the rest: under the smallest scale every element that is not 0 counts
        // as large and is summed in fp64, whatever its magnitude.  A token below the smallest scale is summed in fp64 too.
        const int e = high ? min((int)(high >> 7), (int)(mid >> 7) + 2) + 3 : 0;
        below = high != 0 && e < 15;
        const int se = e < 15 ? 15 : e > 250 ? 250 : e;
#pragma unroll
        for (int j = 0; j < 4; ++j) above += mx[j] > gram_limit(se) ? 1 : 0;
        if ((tid & 3) == 0) {
            sh->scale_exp[r] = se;
            sh->token[r] = tk;
            sh->first[r] = r / m * m;
        }
    }
    fence_proxy_async();
    tc_fence_before();
    const int n_two = __syncthreads_count(above >= 2);
    if (below) sh->fp64 = 1;
    tc_fence_after();
    const uint32_t tmem = sh->tmem_base;
    const int n_steps = (p.d + kGramStep - 1) / kGramStep;
    // this CTA's steps, and how many large elements it may note (formed again where they are needed: registers are what the loop is short of)
    auto step_at = [&](int part) { return (int)((long long)n_steps * part / gp.splits); };
    auto most_noted = [&]() { return min((step_at(rank + 1) - step_at(rank)) * kGramStep, kGramList); };
    // Large elements cost 20 (a dimension that is large in every row) to 70 ns each (one here, one there), the sums in fp64 49 ns per
    // dimension: fp64 from one element per dimension on, or from one scattered one per two dimensions on.  A tile whose samples already
    // show so many goes there directly.  With a share p of the pieces of eight above the bound, two of a thread's four are in 6 p^2 of
    // the 512 threads, and a dimension holds 16 p large elements; pairs are counted because a single dimension that is large in every
    // row must not decide.
    const int s0 = step_at(rank);
    int s1 = step_at(rank + 1);
    {
        const long long dims = (long long)(s1 - s0) * kGramStep, most = most_noted();
        if (n_two * dims * dims > 6LL * kGramProducers * (5 * most / 64) * (5 * most / 64)) {
            s1 = s0;
            sh->fp64 = 1;
        }
    }

    if (warp == kGramProducers / 32) {
        // ================= MMA issuer =================
        if (lane == 0) {
            const uint32_t i_hhm = instr_desc_s8(kGramRows, 256), i_mm = instr_desc_s8(kGramRows, 128), i_c = instr_desc_f16(kGramRows, kGramRows);
            const uint64_t d_rx = smem_desc(smem_u32(ring), 16, 1024, 2), d_dg = smem_desc(smem_u32(digits), 16, 1024, 2);
            RingPos rp{0, 0};
            for (int s = s0; s < s1; ++s, rp.advance(kGramSlots)) {
                if (!gram_wait_limited(sh, hdr, &sh->full[rp.slot], rp.phase, 1)) break;
                tc_fence_after();
                const uint64_t rd = d_rx + (uint64_t)((uint32_t)(rp.slot * 2 * kGramRTile) >> 4), xd = rd + (kGramRTile >> 4);
                const uint64_t hd = d_dg + (uint64_t)((uint32_t)((rp.slot >> 1) * 2 * kGramRTile + (rp.slot & 1) * 64) >> 4), md = hd + (kGramRTile >> 4);
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) {
                    tc_mma_i8(tmem, hd + 2 * ks, hd + 2 * ks, i_hhm, s > s0 || ks ? 1u : 0u);               // <H,H> and <H,M>
                    tc_mma_i8(tmem + 256, md + 2 * ks, md + 2 * ks, i_mm, s > s0 || ks ? 1u : 0u);          // <M,M>
                }
#pragma unroll
                for (int ks = 0; ks < 4; ++ks) tc_mma(tmem + 384, rd + 2 * ks, xd + 2 * ks, i_c, s > s0 || ks ? 1u : 0u);
                tc_commit(smem_u32(&sh->empty[rp.slot]));
            }
            tc_commit(smem_u32(&sh->done));
            gram_wait(sh, hdr, &sh->done, 0, 2, true);     // all tensor-core work is complete before tensor memory is released
        }
    } else {
        // ================= producers: thread = piece (tid & 7) of rows r and r + 64 =================
        // A warp's four rows are r, r + 4, r + 1, r + 5: the 8-byte digit stores of a half warp then fall into different halves of
        // the swizzled 128-byte rows.
        const int piece = lane & 7, sub = lane >> 3;
        const int row0 = (warp >> 1) * 8 + (warp & 1) * 2 + (sub & 1) * 4 + (sub >> 1);
        const uint4 *src[2];                                         // this thread's piece of the round's first step
        uint64_t inv2[2];
        const int s_full = p.d / kGramStep;                          // steps whose every piece exists
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int r = row0 + 64 * i, tk = sh->token[r];
            // a row without a token reads the sequence's first one, scaled by 0; nobody looks at its sums
            src[i] = reinterpret_cast<const uint4 *>(E + (size_t)(tk >= 0 ? tk : p.seq_off[b]) * p.d + piece * 8) + (size_t)s0 * (kGramStep / 8);
            const uint32_t inv = tk >= 0 ? (uint32_t)(127 + kGramUnit - sh->scale_exp[r]) << 23 : 0u;   // 1 / s
            inv2[i] = f2_pack(inv, inv);
        }
        auto load = [&](int s, int ahead, int y) {                   // ahead: steps from the round's first one
            if (s < s_full || (s == s_full && s * kGramStep + piece * 8 < p.d)) return __ldg(src[y] + ahead * (kGramStep / 8));
            return make_uint4(0, 0, 0, 0);
        };
        uint4 buf[kGramAhead][2];
#pragma unroll
        for (int i = 0; i < kGramAhead; ++i)
#pragma unroll
            for (int y = 0; y < 2; ++y) buf[i][y] = load(s0 + i, i, y);
        // byte offsets of this thread's pieces in the tiles: row r + 64 lies 8 KB on, with the same swizzle; the digits' rows hold two
        // steps, the odd step's sixteen-byte chunks are the even one's with bit 2 flipped
        const uint32_t sw = row0 & 7, rt = smem_u32(ring) + row0 * 128 + ((piece ^ sw) << 4);
        const uint32_t dg0 = smem_u32(digits) + row0 * 128 + (((piece >> 1) ^ sw) << 4) + (piece & 1) * 8, dg1 = dg0 ^ 64;
        uint32_t parity = 1;
        for (int sb = s0; sb < s1; sb += kGramSlots, parity ^= 1) {
#pragma unroll
            for (int i = 0; i < kGramSlots; ++i) {                   // step s uses slot i and register buffer i % kGramAhead
                const int s = sb + i;
                if (s >= s1) break;
                gram_wait(sh, hdr, &sh->empty[i], parity, 3);        // after a time-out nobody reads the ring any more
                const uint32_t rts = rt + i * 2 * kGramRTile, dgs = (i & 1 ? dg1 : dg0) + (i >> 1) * 2 * kGramRTile;
#pragma unroll
                for (int y = 0; y < 2; ++y) {
                    uint4 &u = buf[i % kGramAhead][y];
                    GramSplit g = gram_split(u, inv2[y]);
                    if (g.large) {                                                 // something above the bound: take it out, note it
                        u = gram_take_out(sh, u, row0 + 64 * y, s * kGramStep + piece * 8);
                        g = gram_split(u, inv2[y]);
                    }
                    u = load(s + kGramAhead, i + kGramAhead, y);
                    st_shared_v2(dgs + y * 8192, g.h);
                    st_shared_v2(dgs + y * 8192 + kGramRTile, g.m);
                    st_shared_v4(rts + y * 8192, g.r);
                    st_shared_v4(rts + y * 8192 + kGramRTile, g.x);
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(&sh->full[i]));
            }
            src[0] += kGramSlots * (kGramStep / 8);
            src[1] += kGramSlots * (kGramStep / 8);
        }
        gram_wait(sh, hdr, &sh->done, 0, 4);
        __syncwarp();
        // ---- the CTA's block of sums: P[i][a] over the row's own crop, and the products with the same cell one frame on / back;
        //      <x_i, x_j> / (s_i s_j) = P_ij + P_ji
        if (!sh->abort) {
            tc_fence_after();
            const int r = (warp & 3) * 32 + lane, col0 = sh->first[r];
            const uint32_t base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                const int cb = (warp >> 2) * 32 + h * 16;
                float acc[4][16];
#pragma unroll
                for (int k = 0; k < 4; ++k) tmem_ld16(base + k * 128 + cb, acc[k]);
                tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const int col = cb + e, rel = col - col0;
                    const bool in_crop = rel >= 0 && rel < m, next = col == r + m, prev = col == r - m;
                    // formed for every column: a branch per column would put their chains one behind the other (3.2 us)
                    const double v = fma(32768.0, int_to_double(acc[0][e]), fma(256.0, int_to_double(acc[1][e]), 0.5 * (int_to_double(acc[2][e]) + (double)acc[3][e])));
                    if (in_crop) P[r * kGramPStride + rel] = v;
                    if (next) t_next[r] = v;
                    if (prev) t_prev[r] = v;
                }
            }
            tc_fence_before();
        }
    }
    if (gp.part != 1) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __syncthreads();
    if (warp == kGramProducers / 32) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
    bool good = !sh->abort;
    // ---- elements above the bound
    const int n_list = !good ? 0 : sh->fp64 ? kGramList + 1 : sh->n_list;
    if (n_list > 0) {
        const int k0 = step_at(rank) * kGramStep, k1 = step_at(rank + 1) * kGramStep;
        if (n_list > most_noted() || !gram_add_list(sh, ring + kGramScratch, P, E, p.d, m, n_list, (k1 - k0) / 2))
            gram_sum_fp64(sh, reinterpret_cast<double *>(ring + kGramScratch), P, E, p.d, m, k0, min(p.d, k1));
    }
    // ---- the other CTAs' shares of the embedding dimension (same addresses in their shared memory), in rank order
    if (gp.splits > 1) {
        cluster_sync_all();
        if (rank == 0) {
            uint32_t gave_up = 0;                                    // one part missing: no sums at all
            for (int q = 1; q < gp.splits; ++q) gave_up |= ld_cluster_u32(cluster_map(smem_u32((const void *)&sh->abort), (uint32_t)q));
            if (gp.splits == 2) gram_add_peers<2, 9>(P);
            else if (gp.splits == 4) gram_add_peers<4, 3>(P);
            else gram_add_peers<8, 2>(P);
            good = good && gave_up == 0;
        }
        cluster_sync_all();                                          // nobody leaves while its shared memory is read
        if (gp.part == 2) asm volatile("griddepcontrol.wait;" ::: "memory");
        if (rank != 0) return;
    }
    if (gp.part == 2 && gp.splits == 1) asm volatile("griddepcontrol.wait;" ::: "memory");
    const int own_rows = (own_end - f0) * m;
    if (!good) {                                                      // a wait gave up: scores that cannot be taken for any
        if (tid < own_rows && sh->token[tid] >= 0) p.s_spa[sh->token[tid]] = p.tdot[sh->token[tid]] = __longlong_as_double(0x7ff8000000000000ll);
        return;
    }
    __syncthreads();
    // ---- scores: norms, cosines, their variance per row (the shared frame's belong to the next tile)
    if (tid < kGramRows) {
        const int a = tid - sh->first[tid];
        const double n2 = 2.0 * P[tid * kGramPStride + a];
        sh->inv_root[tid] = n2 > 0.0 ? rsqrt(n2) : -1.0;             // also for a norm that is NaN
    }
    __syncthreads();
    if (tid < own_rows && sh->token[tid] >= 0) {
        // The fusion gets the cosine with the next frame itself.  All three sums of a cosine are then this
        // tile's: another tile may have added up other parts of the dimensions, and where frames are equal (a cosine of 1, a variance
        // of 0) the difference of their roundings would be standardised to scores of several sigma.
        const int tk = sh->token[tid], nx = tid + m;
        const double in = sh->inv_root[tid], ix = nx < kGramRows && sh->token[nx] >= 0 ? sh->inv_root[nx] : -1.0;
        if (nx < kGramRows && sh->token[nx] >= 0) p.tdot[tk] = in >= 0.0 && ix >= 0.0 ? (t_next[tid] + t_prev[nx]) * (in * ix) : 0.0;
    }
    for (int i = tid; i < kGramRows * kMaxCrop; i += kGramThreads) {
        const int r = i / kMaxCrop, cj = i % kMaxCrop, fr = sh->first[r], a = r - fr;
        if (cj >= m || cj <= a || fr + cj >= kGramRows) continue;
        // a cosine is 0 unless both norms are above 0: one NaN element must not reach the rest of the crop
        const double ia = sh->inv_root[r], ic = sh->inv_root[fr + cj];
        const double cs = ia >= 0.0 && ic >= 0.0 ? (P[r * kGramPStride + cj] + P[(fr + cj) * kGramPStride + a]) * (ia * ic) : 0.0;
        P[r * kGramPStride + cj] = cs;
        P[(fr + cj) * kGramPStride + a] = cs;
    }
    __syncthreads();
    if (tid < 4 * kGramRows) {                                        // four threads per row
        const int r = tid >> 2, tk = sh->token[r], fr = sh->first[r], a = r - fr;
        int M = m;                                                    // a partial frame holds the first cells of a crop
        while (M > 1 && (fr + M > kGramRows || sh->token[fr + M - 1] < 0)) --M;
        const double *row = P + r * kGramPStride;
        double mu = 0.0, var = 0.0;
        for (int j = tid & 3; j < M; j += 4) mu += j == a ? 1.0 : row[j];
        mu += __shfl_xor_sync(0xffffffffu, mu, 1);
        mu += __shfl_xor_sync(0xffffffffu, mu, 2);
        mu /= M;
        for (int j = tid & 3; j < M; j += 4) {
            const double dv = (j == a ? 1.0 : row[j]) - mu;
            var = fma(dv, dv, var);
        }
        var += __shfl_xor_sync(0xffffffffu, var, 1);
        var += __shfl_xor_sync(0xffffffffu, var, 2);
        if ((tid & 3) == 0 && tk >= 0 && r < own_rows) p.s_spa[tk] = var / M;
    }
}

// How a call is laid out, and about how long its tiles take.
struct GramPlan {
    GramParams gp;
    long long tiles, full;           // all, and those of the first launch where there are two
    int split, split_rest;           // CTAs per tile, and in the second launch
    bool two;
    double cost;                     // us
};
static int32_t gram_plan(const SelectParams &p, GramPlan &plan) {
    static PerDeviceOnce attr_set;
    static std::atomic<int> cluster_room_of[kMaxDevices][3];         // clusters of 2, 4, 8 that are resident together
    int dev;
    if (attr_set.needed(dev)) {
        HIPPO_CUDA_TRY(cudaFuncSetAttribute(select_gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGramSmemBytes));
        for (int i = 0; i < 3; ++i) {
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = 2u << i;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(2u << i);
            cfg.blockDim = dim3(kGramThreads);
            cfg.dynamicSmemBytes = kGramSmemBytes;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int n = 0;
            if (cudaOccupancyMaxActiveClusters(&n, select_gram_kernel, &cfg) != cudaSuccess) { (void)cudaGetLastError(); n = 1; }
            cluster_room_of[dev < 0 ? 0 : dev][i].store(n < 1 ? 1 : n, std::memory_order_relaxed);
        }
        attr_set.mark(dev);
    }
    const std::atomic<int> *cluster_room = cluster_room_of[dev < 0 ? 0 : dev];
    GramParams &gp = plan.gp;
    const int fy = p.grid_h / p.crop_h, fx = p.grid_w / p.crop_w, ey = p.grid_h % p.crop_h, ex = p.grid_w % p.crop_w;
    for (int i = 0; i < 4; ++i) {
        GramClass &c = gp.cls[i];
        const bool by = (i & 2) != 0, bx = (i & 1) != 0;
        c.h = by ? ey : p.crop_h;
        c.w = bx ? ex : p.crop_w;
        c.n_y = by ? (ey ? 1 : 0) : fy;
        c.n_x = bx ? (ex ? 1 : 0) : fx;
        c.y0 = by ? fy * p.crop_h : 0;
        c.x0 = bx ? fx * p.crop_w : 0;
        if (c.n_y * c.n_x == 0) { c.n_y = c.n_x = 0; c.h = c.w = 1; }
        c.frames = kGramRows / (c.h * c.w);
    }
    long long tiles = 0, live = 0;                                   // live: with a token at all
    for (int b = 0; b < p.batch; ++b) {
        gp.tile_off[b] = (int)tiles;
        const int n_frames = p.frame_off[b + 1] - p.frame_off[b], n_v = p.seq_off[b + 1] - p.seq_off[b];
        for (int i = 0; i < 4; ++i) tiles += (long long)gp.cls[i].n_y * gp.cls[i].n_x * gram_class_tiles(n_frames, gp.cls[i].frames);
        if (n_frames > 1) { live += tiles - gp.tile_off[b]; continue; }
        for (int y = 0; y < p.grid_h; y += p.crop_h)
            for (int x = 0; x < p.grid_w; x += p.crop_w) live += y * p.grid_w + x < n_v ? 1 : 0;
    }
    for (int b = p.batch; b <= kSelMaxBatch; ++b) gp.tile_off[b] = (int)tiles;
    // CTAs per tile: a step takes about 0.85 us, a CTA 12 us besides, the meeting of a cluster 3.  Not every SM can be part of a
    // cluster (16 clusters of 8 ran in two waves), so the room for each size is asked for.
    const int n_steps = ceil_div(p.d, kGramStep);
    auto best_split = [&](long long n, int &split) {
        double best_cost = 1e30;
        for (int s = 1; s <= 8 && s <= n_steps; s *= 2) {
            const long long room = s == 1 ? kNumSMs : cluster_room[s == 2 ? 0 : s == 4 ? 1 : 2].load(std::memory_order_relaxed);
            const double cost = (double)((n + room - 1) / room) * (0.85 * ceil_div(n_steps, s) + 12.0 + (s > 1 ? 3.0 : 0.0));
            if (cost < best_cost) { best_cost = cost; split = s; }
        }
        return best_cost;
    };
    // Several waves: the last, partly filled one is a launch of its own with more CTAs per tile (65,536 tokens of 8,192: 645 tiles
    // are 4.4 waves).
    plan.tiles = tiles;
    plan.full = tiles / kNumSMs * kNumSMs;
    plan.cost = best_split(live, plan.split);
    plan.cost += 2.0 * (tiles - live) * plan.split / kNumSMs;        // CTAs that find nothing and leave
    plan.split_rest = 1;
    plan.two = false;
    if (live == tiles && plan.full > 0 && plan.full < tiles) {
        const double cost = plan.full / kNumSMs * (0.85 * n_steps + 12.0) + best_split(tiles - plan.full, plan.split_rest);
        plan.two = cost < 0.98 * plan.cost;
        if (plan.two) plan.cost = cost;
    }
    return HIPPO_OK;
}

int32_t select_gram_cost(const SelectParams &p, double &us) {
    GramPlan plan;
    const int32_t rc = gram_plan(p, plan);
    us = rc == HIPPO_OK ? plan.cost : 0.0;
    return rc;
}

int32_t launch_select_gram(const SelectParams &p, WsHeader *header, cudaStream_t stream) {
    GramPlan plan;
    const int32_t rc = gram_plan(p, plan);
    if (rc != HIPPO_OK) return rc;
    GramParams &gp = plan.gp;
    gp.header = header;
    for (int part = plan.two ? 1 : 0; part <= (plan.two ? 2 : 0); ++part) {
        gp.part = part;
        gp.tile0 = part == 2 ? (int)plan.full : 0;
        gp.splits = part == 0 ? plan.split : part == 1 ? 1 : plan.split_rest;
        const long long n = part == 0 ? plan.tiles : part == 1 ? plan.full : plan.tiles - plan.full;
        cudaLaunchAttribute attr[2];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = (unsigned)gp.splits;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(n * gp.splits));
        cfg.blockDim = dim3(kGramThreads);
        cfg.dynamicSmemBytes = kGramSmemBytes;
        cfg.stream = stream;
        cfg.attrs = attr;
        cfg.numAttrs = gp.splits > 1 ? 2 : 1;
        HIPPO_CUDA_TRY(cudaLaunchKernelEx(&cfg, select_gram_kernel, p, gp));
        count_launches(1);
    }
    return HIPPO_OK;
}

}  // namespace hippo
