// hippo_accept: lossless speculative acceptance (Section 3.2, Eq. 1 and the resampling rule that follows it).
//
//   P_j, Q_j = softmax(target row j), softmax(draft row j)            (temperature 1)
//   accept x_{j+1} iff u_accept[j] * Q_j[x] < P_j[x]                   (probability min(1, P/Q), Eq. 1)
//   first rejection at n < gamma: draw from norm(max(0, P_n - Q_n));   none: draw the bonus token from P_gamma
//   draw = inverse CDF in ascending token id: smallest t with cumsum_t > u_resample * total
//
// All probabilities, normalisers and CDFs are fp64 so that the decisions agree with an fp64 reference unless a
// uniform lands within ~1e-15 of a boundary.  Three kernels over the vocabulary, chained with programmatic
// dependent launches (each waits for its predecessor before it reads anything):
//   stats   per (sequence, logit row, 4096-token chunk): max and sum of exponentials
//   weigh   per (sequence, piece: a chunk, or a quarter of one where that still fits one wave): every CTA merges the
//           chunk stats of its sequence and runs the accept tests itself (a few hundred values; cheaper than a launch
//           of its own), then scans the residual (or bonus) weights of its piece in token order and stores the
//           running sum after every 16 tokens
//   pick    per sequence: locate the piece, then the 16-token group, then the token where the CDF crosses
//           u * total; only that one group's weights are evaluated again
#include <math.h>

#include <atomic>
#include <mutex>

#include "common.cuh"

namespace hippo {

// The steps are bound by the latency of fp64 exponentials until there is a wave of chunks: a chunk goes to 1,024 threads of four
// tokens, or to fewer with more (see the launches).
constexpr int kAccThreads = 1024;
constexpr int kAccWarps = kAccThreads / 32;
constexpr int kAccPerThread = 4;
constexpr int kAccChunk = kAccThreads * kAccPerThread;  // 4096 vocabulary entries per chunk
constexpr int kAccGroup = 16;                           // tokens per stored running sum
constexpr int kAccGroups = kAccChunk / kAccGroup;
constexpr int kAccMaxRows = 2 * 64 + 1;
constexpr bool kAcceptFusedByDefault = false;

struct RowInfo {
    double Mp, Zp, Mq, Zq;  // max logit and 1 / (sum of exponentials) of target row n / draft row n
    int32_t n;              // accepted count
    int32_t bonus;          // 1: n == gamma, draw from P_gamma
    int32_t pad[2];
};

struct AcceptParams {
    const float *tl, *dl, *ua, *ur;
    const int32_t *x;
    int32_t *n_acc, *out;
    double2 *stats;  // [B][2*gamma+1][n_chunks]: (max, sum exp)
    double *tscan;   // [B][n_chunks][kAccGroups]: running sum of the weights, within a piece, after each group of 16 tokens
    RowInfo *info;   // [B]
    int B, gamma, V, n_chunks;
    int piece;       // tokens that a CTA of the weigh step takes
};

__device__ __forceinline__ const float *logit_row(const AcceptParams &p, int b, int r) {
    // r in [0, gamma]: target row r; r in (gamma, 2*gamma]: draft row r - gamma - 1
    return r <= p.gamma ? p.tl + ((size_t)b * (p.gamma + 1) + r) * p.V : p.dl + ((size_t)b * p.gamma + (r - p.gamma - 1)) * p.V;
}

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// In-order inclusive scan over the warp's lanes.
__device__ __forceinline__ double warp_scan_inclusive(double v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// In-order inclusive scan over the block's threads (thread i holds element i).  Deterministic; *total is the last thread's sum,
// *before the sum in front of the thread.
template <int T>
__device__ __forceinline__ double block_scan_inclusive(double v, double *warp_tot /* [32] shared */, double *total, double *before = nullptr) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    v = warp_scan_inclusive(v);
    __syncthreads();  // protect warp_tot from a previous use
    if (lane == 31) warp_tot[warp] = v;
    __syncthreads();
    const double t = warp_scan_inclusive(lane < T / 32 ? warp_tot[lane] : 0.0);
    const double pre = __shfl_sync(0xffffffffu, t, warp ? warp - 1 : 0);
    *total = __shfl_sync(0xffffffffu, t, T / 32 - 1);
    if (before) {
        const double left = __shfl_up_sync(0xffffffffu, v, 1);
        *before = (warp ? pre : 0.0) + (lane ? left : 0.0);
    }
    return warp ? v + pre : v;
}

// The statistics are bound by the issue of their exponentials, 2 * gamma + 1 rows of them in fp64.  exp(x), -709 < x <= 0 or NaN, by table and
// polynomial (P. T. P. Tang, "Table-driven implementation of the exponential function in IEEE floating-point arithmetic", ACM TOMS 15,
// 1989): x = (64 e + j) ln 2 / 64 + r, |r| <= h = ln 2 / 128, exp(x) = 2^e 2^(j/64) (1 + r + ... + r^5 / 120).  The first term left out, r^6 / 720,
// is put back but for a 32nd of itself by its Chebyshev expansion, r^6 = 3/2 h^2 r^4 - 9/16 h^4 r^2 + h^6 / 32 + ..., in the factors of r^4 and
// r^2.  Error, over 10^8 arguments: 0.53 ulp at most, 0.250 on average; the series as it stands 0.82 and 0.254, exp() 0.88 and 0.258.
// The table holds 2^(j/64), its upper word less j << 14 so that adding k << 14, k = 64 e + j, adds e to the exponent, and the relative
// error of its rounding; in eight copies so that the lanes of a quarter warp read different banks.  Statistics at batch 8, gamma 7,
// vocabulary 152,064: 31 us with exp(), its branch taken out and the checks in double; 26 us now.
constexpr int kAccExpSize = 64, kAccExpCopies = 8;
__device__ const double2 kAccExp2[kAccExpSize] = {
    {1.0, 0}, {1.0108892860517005, -1.50706698e-17}, {1.0218971486541166, 4.99974487e-17}, {1.0330248790212284, 7.35784687e-18},
    {1.0442737824274138, 8.18931764e-17}, {1.0556451783605572, 1.66658814e-18}, {1.0671404006768237, -7.40282531e-17}, {1.0787607977571199, -6.17065475e-17},
    {1.0905077326652577, -2.79391149e-17}, {1.102382583307841, 4.77695943e-17}, {1.1143867425958924, 9.34171061e-17}, {1.1265216186082418, 4.58567033e-17},
    {1.1387886347566916, 7.82657326e-17}, {1.1511892299529827, 2.82378443e-17}, {1.1637248587775775, 3.29047266e-17}, {1.1763969916502812, 4.72136812e-17},
    {1.189207115002721, 3.34846233e-17}, {1.202156731452703, 5.52755005e-17}, {1.215247359980469, -6.34655211e-17}, {1.22848053610687, -1.54563428e-17},
    {1.241857812073484, 3.7508542e-17}, {1.255380757024691, -5.34609901e-18}, {1.2690509571917332, 2.10230497e-18}, {1.2828700160787783, 1.33575101e-17},
    {1.2968395546510096, 1.95725853e-17}, {1.3109612115247644, -5.47806912e-17}, {1.3252366431597413, -2.15714773e-17}, {1.339667524053303, 6.66380459e-17},
    {1.3542555469368927, 5.68648096e-17}, {1.3690024229745905, 7.00787505e-17}, {1.383909881963832, -4.89230675e-17}, {1.3989796725383112, -6.87230372e-17},
    {1.4142135623730951, -6.83580866e-17}, {1.42961333839197, -8.41601163e-18}, {1.4451808069770467, -2.09230438e-17}, {1.460917794180647, -3.83346497e-17},
    {1.4768261459394993, -2.35910948e-17}, {1.4929077282912648, 9.5068971e-18}, {1.5091644275934228, -6.73521923e-17}, {1.5255981507445384, -7.22663547e-17},
    {1.5422108254079407, 5.15483012e-17}, {1.559004400237837, 2.42539858e-17}, {1.5759808451078865, -6.43213178e-18}, {1.593142151342267, -6.33616186e-17},
    {1.6104903319492543, 1.53414101e-17}, {1.6280274218573478, -4.12336733e-17}, {1.645755478153965, -6.15260289e-17}, {1.6636765803267364, 3.54094826e-17},
    {1.681792830507429, 4.87516053e-17}, {1.7001063537185235, -4.71953966e-18}, {1.718619298122478, -1.07724871e-17}, {1.7373338352737062, 1.82140544e-17},
    {1.7562521603732995, 1.68548729e-17}, {1.7753764925265212, 3.62161594e-17}, {1.7947090750031072, 1.0156219e-17}, {1.8142521755003989, -5.49511897e-17},
    {1.8340080864093424, 1.79012691e-17}, {1.8539791250833855, 5.26537077e-17}, {1.8741676341103, -3.2669241e-17}, {1.8945759815869656, 1.79639327e-17},
    {1.9152065613971474, -5.54506562e-17}, {1.9360617934922943, 5.33680588e-17}, {1.9571441241754002, 4.57849153e-17}, {1.978456026387951, 2.04142789e-17},
};
template <int T>
__device__ __forceinline__ void acc_exp_table(double2 *tab) {
    for (int i = threadIdx.x; i < kAccExpSize * kAccExpCopies; i += T) {
        const int j = i / kAccExpCopies;
        const double2 v = kAccExp2[j];
        tab[i] = make_double2(__hiloint2double(__double2hiint(v.x) - (j << 14), __double2loint(v.x)), v.y);
    }
}
__device__ __forceinline__ double acc_exp(double x, const double2 *tab /* this lane's copy */) {
    const double round = 6755399441055744.0;               // 1.5 * 2^52
    const double t = fma(x, 92.33248261689366, round);     // 64 / ln 2
    const int k = __double2loint(t);
    const double n = t - round;
    double r = fma(n, -0.010830424695996044, x);           // ln 2 / 64: the upper 34 bits, the rest
    r = fma(n, -2.5310172166650877e-13, r);
    double q = fma(r, 1.0 / 120.0, 0.04166672775942661);   // 1 / 24 + h^2 / 480
    q = fma(r, q, 1.0 / 6.0);
    q = fma(r, q, 0.4999999999993282);                     // 1 / 2 - h^4 / 1280
    const double2 s = tab[(k & (kAccExpSize - 1)) * kAccExpCopies];
    q = fma(r * r, q, r + s.y);
    const double p = __hiloint2double(__double2hiint(s.x) + (k << 14), __double2loint(s.x));
    return fma(p, q, p);
}
// Max and sum of exponentials of one 4096-token chunk of one logit row, by T threads.  `tab`: this lane's copy of the table.
template <int T>
__device__ __forceinline__ void stats_item(const AcceptParams &p, int b, int r, int c, const double2 *tab) {
    constexpr int kPer = kAccChunk / T, kWarps = T / 32;
    __shared__ float smax[kWarps];
    __shared__ double ssum[kWarps];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __syncthreads();   // the shared arrays may still be read by the previous item
    const float *row = logit_row(p, b, r);
    float v[kPer];
    if ((c + 1) * kAccChunk <= p.V && (((uintptr_t)row) & 15) == 0 && (p.V & 3) == 0) {      // full chunk, 16-byte aligned
#pragma unroll
        for (int e = 0; e < kPer; e += 4) {
            const float4 t = __ldg(reinterpret_cast<const float4 *>(row + c * kAccChunk) + (e / 4) * T + tid);
            v[e] = t.x; v[e + 1] = t.y; v[e + 2] = t.z; v[e + 3] = t.w;
        }
    } else {
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
            const int t = c * kAccChunk + e * T + tid;
            v[e] = t < p.V ? row[t] : -INFINITY;
        }
    }
    float m = -INFINITY;      // not v[0]: a chunk of nothing but NaN has this maximum and stays out of its row's sum
#pragma unroll
    for (int e = 0; e < kPer; ++e) m = fmaxf(m, v[e]);
#pragma unroll
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) smax[warp] = m;
    __syncthreads();
    m = smax[lane % kWarps];
#pragma unroll
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    // An element 700 below the maximum or lower counts as one 700 below (its upper word is limited to that of -700): 1e-304 does not reach a
    // sum that is 1 at least (where the maximum itself is -inf nobody looks at the sum).  NaN, inf - inf too, makes NaN of the sum.
    const double md = (double)m;
    double s = 0.0;
    bool nan = m == INFINITY;
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
        const double x = (double)v[e] - md;
        s += acc_exp(__hiloint2double((int)min((unsigned)__double2hiint(x), 0xC085E000u), __double2loint(x)), tab);
        nan |= isnan(v[e]);
    }
    if (nan) s = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) ssum[warp] = s;
    __syncthreads();
    if (warp == 0) {
        s = lane < kWarps ? ssum[lane] : 0.0;
#pragma unroll
        for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) p.stats[((size_t)b * (2 * p.gamma + 1) + r) * p.n_chunks + c] = make_double2((double)m, s);
    }
}

template <int T>
__global__ void __launch_bounds__(T) accept_stats_kernel(const AcceptParams p) {
    __shared__ double2 tab[kAccExpSize * kAccExpCopies];
    acc_exp_table<T>(tab);
    pdl_wait();
    pdl_trigger();
    stats_item<T>(p, blockIdx.z, blockIdx.y, blockIdx.x, tab + (threadIdx.x & (kAccExpCopies - 1)));    // begins with a barrier
}

// Weight of token t in the distribution the emitted token is drawn from.  use_target_only: bonus row, or the
// degenerate rejection with P_n == Q_n everywhere.
__device__ __forceinline__ double weight_of(float tl, float dl, const RowInfo &ri, bool use_target_only) {
    const double P = exp((double)tl - ri.Mp) * ri.Zp;
    if (use_target_only) return P;
    const double Q = exp((double)dl - ri.Mq) * ri.Zq;
    const double w = P - Q;
    return w > 0.0 ? w : 0.0;
}
__device__ __forceinline__ double draw_weight(const float *trow, const float *drow, int t, const RowInfo &ri, bool use_target_only) {
    return weight_of(trow[t], use_target_only ? 0.f : drow[t], ri, use_target_only);
}

// Thread-local weights of piece c (T threads, kPer consecutive tokens each) and their in-order sum.
template <int T, int kPer>
__device__ __forceinline__ double chunk_local(const float *trow, const float *drow, int c, int V, const RowInfo &ri,
                                              bool target_only, double *w) {
    double s = 0.0;
    const int t0 = (c * T + (int)threadIdx.x) * kPer;
    float tv[kPer], dv[kPer];
    const bool vec = t0 + kPer <= V && (((uintptr_t)(trow + t0) | (target_only ? 0 : (uintptr_t)(drow + t0))) & (kPer >= 4 ? 15 : 7)) == 0;
    if (vec && kPer == 2) {
        const float2 a = __ldg(reinterpret_cast<const float2 *>(trow + t0));
        float2 d = make_float2(0.f, 0.f);
        if (!target_only) d = __ldg(reinterpret_cast<const float2 *>(drow + t0));
        tv[0] = a.x; tv[1] = a.y;
        dv[0] = d.x; dv[1] = d.y;
    } else if (vec) {
#pragma unroll
        for (int e = 0; e + 3 < kPer; e += 4) {
            const float4 a = __ldg(reinterpret_cast<const float4 *>(trow + t0 + e));
            float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
            if (!target_only) d = __ldg(reinterpret_cast<const float4 *>(drow + t0 + e));
            tv[e] = a.x; tv[e + 1] = a.y; tv[e + 2] = a.z; tv[e + 3] = a.w;
            dv[e] = d.x; dv[e + 1] = d.y; dv[e + 2] = d.z; dv[e + 3] = d.w;
        }
    } else {
#pragma unroll
        for (int e = 0; e < kPer; ++e) {
            const int t = t0 + e;
            tv[e] = t < V ? trow[t] : 0.f;
            dv[e] = (t < V && !target_only) ? drow[t] : 0.f;
        }
    }
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
        w[e] = t0 + e < V ? weight_of(tv[e], dv[e], ri, target_only) : 0.0;
        s += w[e];
    }
    return s;
}

// Merge of the chunk statistics of every logit row of sequence b and the sequential accept tests.  Run by all
// threads of a block; the result is identical in every block of the sequence (same data, same order).
template <int T>
__device__ __forceinline__ RowInfo decide_rows(const AcceptParams &p, int b, double *rowstat /* shared [2*gamma+1][3] */, int *s_n) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_rows = 2 * p.gamma + 1;
    // the first 32 draft tokens' logits are on their way while the statistics are merged
    const int32_t *x = p.x + (size_t)b * p.gamma;
    int tok0 = -1;
    float tl0 = 0.f, dl0 = 0.f, u0 = 0.f;
    if (warp == 0 && lane < p.gamma) {
        tok0 = x[lane];
        u0 = p.ua[(size_t)b * p.gamma + lane];
        if ((unsigned)tok0 < (unsigned)p.V) { tl0 = logit_row(p, b, lane)[tok0]; dl0 = logit_row(p, b, p.gamma + 1 + lane)[tok0]; }
    }
    for (int r = warp; r < n_rows; r += T / 32) {
        const double2 *st = p.stats + ((size_t)b * n_rows + r) * p.n_chunks;
        // two chunks per lane stay in registers, which is all of them up to a vocabulary of 262,144
        const double2 none = make_double2(-INFINITY, 0.0);
        const double2 c0 = lane < p.n_chunks ? st[lane] : none, c1 = lane + 32 < p.n_chunks ? st[lane + 32] : none;
        double M = fmax(c0.x, c1.x);
        for (int c = lane + 64; c < p.n_chunks; c += 32) M = fmax(M, st[c].x);
        for (int o = 16; o; o >>= 1) M = fmax(M, __shfl_xor_sync(0xffffffffu, M, o));
        double Z = c0.x != -INFINITY ? c0.y * exp(c0.x - M) : 0.0;
        if (c1.x != -INFINITY) Z += c1.y * exp(c1.x - M);
        for (int c = lane + 64; c < p.n_chunks; c += 32)
            if (st[c].x != -INFINITY) Z += st[c].y * exp(st[c].x - M);
        for (int o = 16; o; o >>= 1) Z += __shfl_xor_sync(0xffffffffu, Z, o);
        if (lane == 0) { rowstat[3 * r] = M; rowstat[3 * r + 1] = Z; }
    }
    __syncthreads();
    if (warp > 0) {
        for (int r = tid - 32; r < n_rows; r += T - 32) rowstat[3 * r + 2] = 1.0 / rowstat[3 * r + 1];     // meanwhile
    } else {
        // lane j tests draft token j (all loads independent), then the first failing lane is n
        int n = p.gamma;
        for (int j0 = 0; j0 < p.gamma; j0 += 32) {
            const int j = j0 + lane;
            bool accept = true;
            if (j < p.gamma) {
                const int rq = p.gamma + 1 + j, tok = j0 ? x[j] : tok0;
                // a token id outside the vocabulary (a fault upstream) is never looked up: it counts as rejected
                accept = false;
                if ((unsigned)tok < (unsigned)p.V) {
                    const float tl = j0 ? logit_row(p, b, j)[tok] : tl0, dl = j0 ? logit_row(p, b, rq)[tok] : dl0;
                    const double P = exp((double)tl - rowstat[3 * j]) / rowstat[3 * j + 1];
                    const double Q = exp((double)dl - rowstat[3 * rq]) / rowstat[3 * rq + 1];
                    const double u = (double)(j0 ? p.ua[(size_t)b * p.gamma + j] : u0);
                    accept = u * Q < P;
                }
            }
            const unsigned rejected = __ballot_sync(0xffffffffu, !accept);
            if (rejected) { n = j0 + __ffs(rejected) - 1; break; }
        }
        if (lane == 0) *s_n = n;
    }
    __syncthreads();
    RowInfo ri;
    ri.n = *s_n;
    ri.bonus = (ri.n == p.gamma);
    ri.Mp = rowstat[3 * ri.n]; ri.Zp = rowstat[3 * ri.n + 2];
    if (ri.n < p.gamma) { ri.Mq = rowstat[3 * (p.gamma + 1 + ri.n)]; ri.Zq = rowstat[3 * (p.gamma + 1 + ri.n) + 2]; }
    else { ri.Mq = 0.0; ri.Zq = 1.0; }
    ri.pad[0] = ri.pad[1] = 0;
    return ri;
}

// Residual (or bonus) weights of one piece of sequence b, scanned in token order.  Every caller re-derives the row
// normalisers and the accept decisions of the sequence (same data, same order: identical everywhere).
template <int T, int kPer>
__device__ __forceinline__ void weigh_item(const AcceptParams &p, int b, int c) {
    __shared__ double rowstat[3 * kAccMaxRows];
    __shared__ double warp_tot[kAccWarps];
    __shared__ int s_n;
    const int tid = threadIdx.x;
    __syncthreads();   // the shared arrays may still be read by the previous item
    const RowInfo ri = decide_rows<T>(p, b, rowstat, &s_n);
    if (c == 0 && tid == 0) {
        const int32_t *x = p.x + (size_t)b * p.gamma;
        int32_t *out = p.out + (size_t)b * (p.gamma + 1);
        for (int j = 0; j < ri.n; ++j) out[j] = x[j];
        for (int j = ri.n; j <= p.gamma; ++j) out[j] = -1;  // out[n] is filled by the pick step
        p.n_acc[b] = ri.n;
        p.info[b] = ri;
    }
    const float *trow = logit_row(p, b, ri.n);
    const float *drow = ri.bonus ? nullptr : logit_row(p, b, p.gamma + 1 + ri.n);
    constexpr int kPerGroup = kAccGroup / kPer;                           // threads that share a group
    double w[kPer], total;
    const double s = chunk_local<T, kPer>(trow, drow, c, p.V, ri, ri.bonus != 0, w);
    const double incl = block_scan_inclusive<T>(s, warp_tot, &total);
    if (tid % kPerGroup == kPerGroup - 1) p.tscan[(size_t)b * p.n_chunks * kAccGroups + (size_t)c * (T * kPer / kAccGroup) + tid / kPerGroup] = incl;
}

template <int T, int kPer>
__global__ void __launch_bounds__(T) accept_weigh_kernel(const AcceptParams p) {
    pdl_wait();
    pdl_trigger();
    weigh_item<T, kPer>(p, blockIdx.y, blockIdx.x);
}

// The emitted token of sequence b: piece, 16-token group and token where the CDF crosses u * total.  ws: the pieces' weights, in shared
// memory.
__device__ __forceinline__ void pick_item(const AcceptParams &p, int b, double *ws) {
    __shared__ double warp_tot[kAccWarps];
    __shared__ double s_prefix, s_target;
    __shared__ int s_chunk, s_tok, s_first;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __syncthreads();   // the shared arrays may still be read by the previous item
    const RowInfo ri = p.info[b];
    const float *trow = logit_row(p, b, ri.n);
    const float *drow = ri.bonus ? nullptr : logit_row(p, b, p.gamma + 1 + ri.n);
    const int groups = p.piece / kAccGroup;       // per piece; the running sum after the last one is the piece's weight
    const double *tscan = p.tscan + (size_t)b * p.n_chunks * kAccGroups;
    const double u = (double)p.ur[b];
    int units = (p.V + p.piece - 1) / p.piece;
    for (int c = tid; c < units; c += kAccThreads) ws[c] = tscan[(size_t)(c + 1) * groups - 1];
    if (tid == 0) { s_chunk = 0x7fffffff; s_tok = 0x7fffffff; s_first = 0x7fffffff; }
    __syncthreads();
    // running sum of the pieces, 1,024 at a time; v, before: this thread's piece of the last batch
    double v = 0.0, before = 0.0, w[kAccPerThread], total;
    auto scan_units = [&](int c0, double cum) {
        v = c0 + tid < units ? ws[c0 + tid] : 0.0;
        block_scan_inclusive<kAccThreads>(v, warp_tot, &total, &before);
        before += cum;
        return cum + total;
    };
    auto total_weight = [&]() {
        double Z = 0.0;
        for (int c0 = 0; c0 < units; c0 += kAccThreads) Z = scan_units(c0, Z);
        return Z;
    };
    double Z = total_weight();
    const bool target_only = ri.bonus || !(Z > 0.0);
    if (target_only && !ri.bonus) {
        // residual is identically zero (P_n == Q_n): fall back to P_n; recompute the totals, by whole chunks
        units = p.n_chunks;
        __syncthreads();
        for (int c = 0; c < units; ++c) {
            const double s = chunk_local<kAccThreads, kAccPerThread>(trow, drow, c, p.V, ri, true, w);
            const double incl = block_scan_inclusive<kAccThreads>(s, warp_tot, &total);
            if (tid == kAccThreads - 1) ws[c] = incl;
        }
        __syncthreads();
        Z = total_weight();
    }
    const double target = u * Z;
    double cum = 0.0;
    for (int c0 = 0; c0 < units; c0 += kAccThreads) {
        if (units > kAccThreads) cum = scan_units(c0, cum);
        const unsigned over = __ballot_sync(0xffffffffu, c0 + tid < units && before + v > target);
        if (over && lane == __ffs(over) - 1) atomicMin(&s_chunk, c0 + tid);
        __syncthreads();
        if (s_chunk != 0x7fffffff) {
            if (s_chunk == c0 + tid) { s_prefix = before; s_target = target; }
            break;
        }
    }
    __syncthreads();
    int tok = -1;
    const int c = s_chunk == 0x7fffffff ? -1 : s_chunk;
    if (c >= 0 && !(target_only && !ri.bonus)) {
        // the 16-token group: the first of the piece whose stored running sum exceeds the target
        const double *scan = tscan + (size_t)c * groups;
        if (tid < groups) {                                            // a multiple of a warp
            const unsigned over = __ballot_sync(0xffffffffu, s_prefix + scan[tid] > s_target);
            if (over && lane == __ffs(over) - 1) atomicMin(&s_first, tid);
        }
        __syncthreads();
        const int first = s_first;
        if (warp == 0 && first != 0x7fffffff) {
            // its tokens, a lane each, in order from the running sum before them
            const int t = c * p.piece + first * kAccGroup + lane;
            const bool in = lane < kAccGroup && t < p.V;
            const double wt = in ? draw_weight(trow, drow, t, ri, target_only) : 0.0;
            const double run = s_prefix + (first ? scan[first - 1] : 0.0) + warp_scan_inclusive(wt);
            const unsigned over = __ballot_sync(0xffffffffu, in && run > s_target), positive = __ballot_sync(0xffffffffu, in && wt > 0.0);
            // rounding may leave the crossing just past the group's end: then its last positive weight
            const int at = over ? __ffs(over) - 1 : positive ? 31 - __clz(positive) : -1;
            if (at >= 0) tok = c * p.piece + first * kAccGroup + at;
        }
    } else if (c >= 0) {
        const double s = chunk_local<kAccThreads, kAccPerThread>(trow, drow, c, p.V, ri, target_only, w);
        const double incl = block_scan_inclusive<kAccThreads>(s, warp_tot, &total);
        double run = s_prefix + (incl - s);  // CDF just before this thread's first token
        int mine = 0x7fffffff;
#pragma unroll
        for (int e = 0; e < kAccPerThread; ++e) {
            run += w[e];
            if (mine == 0x7fffffff && run > s_target) mine = c * kAccChunk + tid * kAccPerThread + e;
        }
        if (mine != 0x7fffffff) atomicMin(&s_tok, mine);
        __syncthreads();
        if (s_tok != 0x7fffffff) tok = s_tok;
    }
    if (tok < 0 && tid == 0) {
        // the CDF never exceeded the target (possible only through rounding): last token with positive weight
        for (int t = p.V - 1; t >= 0; --t)
            if (draw_weight(trow, drow, t, ri, target_only) > 0.0) { tok = t; break; }
    }
    if (tid == 0) p.out[(size_t)b * (p.gamma + 1) + ri.n] = tok;
}

__global__ void __launch_bounds__(kAccThreads) accept_pick_kernel(const AcceptParams p) {
    extern __shared__ double ws[];   // the pieces' weights
    pdl_wait();
    pdl_trigger();
    pick_item(p, blockIdx.x, ws);
}

// ---- the same three steps in one launch ----------------------------------------------------------------------------
// A grid of at most one wave of CTAs walks the items of each step; between the steps all CTAs meet at a counter in the
// workspace header (zeroed before the launch).  The wait at the counter is bounded: after 2 s a CTA records
// HIPPO_ERR_TIMEOUT in the header and leaves, and so does every CTA that sees the status word set.
constexpr unsigned long long kAccWaitLimitNs = 2000000000ull;

__device__ bool accept_grid_barrier(WsHeader *hdr, int which) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int *counter = &hdr->pad[which];
        __threadfence();
        atomicAdd(counter, 1);
        bool ok = true;
        unsigned long long t0 = 0;
        for (;;) {
            int seen;
            asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(seen) : "l"(counter) : "memory");
            if (seen >= (int)gridDim.x) break;
            if (*reinterpret_cast<volatile int *>(&hdr->status) != 0) { ok = false; break; }
            unsigned long long now;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
            if (t0 == 0) t0 = now;
            if (now - t0 > kAccWaitLimitNs) {
                if (atomicCAS(&hdr->status, 0, (int)HIPPO_ERR_TIMEOUT) == 0) hdr->where = 200 + which;
                ok = false;
                break;
            }
            __nanosleep(64);
        }
        s_ok = ok ? 1 : 0;
    }
    __syncthreads();
    return s_ok != 0;
}

__global__ void __launch_bounds__(kAccThreads) accept_fused_kernel(const AcceptParams p, WsHeader *hdr) {
    extern __shared__ double ws[];   // the pieces' weights
    __shared__ double2 tab[kAccExpSize * kAccExpCopies];
    acc_exp_table<kAccThreads>(tab);
    pdl_wait();
    pdl_trigger();
    const int rows = 2 * p.gamma + 1;
    for (int i = blockIdx.x; i < p.B * rows * p.n_chunks; i += gridDim.x)
        stats_item<kAccThreads>(p, i / (rows * p.n_chunks), (i / p.n_chunks) % rows, i % p.n_chunks, tab + (threadIdx.x & (kAccExpCopies - 1)));
    if (!accept_grid_barrier(hdr, 0)) return;
    for (int i = blockIdx.x; i < p.B * p.n_chunks; i += gridDim.x) weigh_item<kAccThreads, kAccPerThread>(p, i / p.n_chunks, i % p.n_chunks);
    if (!accept_grid_barrier(hdr, 1)) return;
    for (int b = blockIdx.x; b < p.B; b += gridDim.x) pick_item(p, b, ws);
}

struct AcceptWs { size_t stats_off, info_off, tscan_off, total; int n_chunks; };
static AcceptWs accept_ws(int B, int gamma, int V) {
    AcceptWs w;
    w.n_chunks = ceil_div(V, kAccChunk);
    w.stats_off = kWsHeaderBytes;
    w.info_off = w.stats_off + align_up((size_t)B * (2 * gamma + 1) * w.n_chunks * sizeof(double2), 256);
    w.tscan_off = w.info_off + align_up((size_t)B * sizeof(RowInfo), 256);
    w.total = w.tscan_off + align_up((size_t)B * w.n_chunks * kAccGroups * sizeof(double), 256);
    return w;
}

// ---- greedy verification (the decoding mode of the paper's experiments): keep draft tokens while they equal the
// arg-max of the target row, then emit the target's arg-max (lowest token id on ties).
//   argmax  per (sequence, target row, chunk): maximum and its first position -> stats[b][row][chunk] = (max, index)
//   greedy  per sequence: merge the chunks of every row, compare with the draft tokens, write the outputs
template <int T>
__global__ void __launch_bounds__(T) accept_argmax_kernel(const AcceptParams p) {
    __shared__ float smax[T / 32];
    __shared__ int sidx[T / 32];
    pdl_wait();
    pdl_trigger();
    const int c = blockIdx.x, r = blockIdx.y, b = blockIdx.z, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float *row = logit_row(p, b, r);
    float m = -INFINITY;
    int mi = 0x7fffffff;
#pragma unroll
    for (int e = 0; e < kAccChunk / T; ++e) {
        const int t = c * kAccChunk + e * T + tid;     // ascending in e: a strict '>' keeps the first maximum
        const float v = t < p.V ? row[t] : -INFINITY;
        if (v > m || (v == m && t < mi && t < p.V)) { m = v; mi = t; }
    }
    for (int o = 16; o; o >>= 1) {
        const float om = __shfl_xor_sync(0xffffffffu, m, o);
        const int oi = __shfl_xor_sync(0xffffffffu, mi, o);
        if (om > m || (om == m && oi < mi)) { m = om; mi = oi; }
    }
    if (lane == 0) { smax[warp] = m; sidx[warp] = mi; }
    __syncthreads();
    if (warp == 0) {
        m = smax[lane % (T / 32)]; mi = sidx[lane % (T / 32)];
        for (int o = 16; o; o >>= 1) {
            const float om = __shfl_xor_sync(0xffffffffu, m, o);
            const int oi = __shfl_xor_sync(0xffffffffu, mi, o);
            if (om > m || (om == m && oi < mi)) { m = om; mi = oi; }
        }
        if (lane == 0) p.stats[((size_t)b * (2 * p.gamma + 1) + r) * p.n_chunks + c] = make_double2((double)m, (double)mi);
    }
}

__global__ void __launch_bounds__(kAccThreads) accept_greedy_kernel(const AcceptParams p) {
    __shared__ int best[kAccMaxRows];
    pdl_wait();
    pdl_trigger();
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_rows = 2 * p.gamma + 1;
    for (int r = warp; r <= p.gamma; r += blockDim.x >> 5) {
        const double2 *st = p.stats + ((size_t)b * n_rows + r) * p.n_chunks;
        double m = -INFINITY, mi = 2147483647.0;
        for (int c = lane; c < p.n_chunks; c += 32)
            if (st[c].x > m || (st[c].x == m && st[c].y < mi)) { m = st[c].x; mi = st[c].y; }
        for (int o = 16; o; o >>= 1) {
            const double om = __shfl_xor_sync(0xffffffffu, m, o), oi = __shfl_xor_sync(0xffffffffu, mi, o);
            if (om > m || (om == m && oi < mi)) { m = om; mi = oi; }
        }
        if (lane == 0) best[r] = (int)mi;
    }
    __syncthreads();
    if (tid == 0) {
        const int32_t *x = p.x + (size_t)b * p.gamma;
        int32_t *out = p.out + (size_t)b * (p.gamma + 1);
        int n = 0;
        while (n < p.gamma && x[n] == best[n]) { out[n] = x[n]; ++n; }
        out[n] = best[n];
        for (int j = n + 1; j <= p.gamma; ++j) out[j] = -1;
        p.n_acc[b] = n;
    }
}

static int32_t launch_accept_greedy(const AcceptParams &p, cudaStream_t s) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kAccThreads);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3((unsigned)p.n_chunks, (unsigned)(p.gamma + 1), (unsigned)p.B);
    if ((long long)p.n_chunks * (p.gamma + 1) * p.B <= 320) {        // as in the sampling mode
        cfg.blockDim = dim3(512);
        HIPPO_CUDA_TRY(cudaLaunchKernelEx(&cfg, accept_argmax_kernel<512>, p));
    } else {
        cfg.blockDim = dim3(256);
        HIPPO_CUDA_TRY(cudaLaunchKernelEx(&cfg, accept_argmax_kernel<256>, p));
    }
    // a warp per row; blocks of 1,024 threads where there are eight rows take 0.5 us longer (batch 64, 300 entries: 6.1 / 5.6 us)
    cfg.blockDim = dim3(p.gamma + 1 <= 8 ? 256 : kAccThreads);
    cfg.gridDim = dim3((unsigned)p.B);
    HIPPO_CUDA_TRY(cudaLaunchKernelEx(&cfg, accept_greedy_kernel, p));
    count_launches(2);
    return HIPPO_OK;
}

// The three kernels, launched with programmatic stream serialization (each one waits before it reads).
static int32_t launch_accept_chain(AcceptParams p, cudaStream_t s) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kAccThreads);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3((unsigned)p.n_chunks, (unsigned)(2 * p.gamma + 1), (unsigned)p.B);
    // Threads per chunk: many while the chunks leave SMs idle (latency), few once there is a wave of them or more (the block's
    // meetings then cost more than they hide).  Vocabulary 152,064, us with 1,024 / 512 / 256 threads for the statistics: batch 1
    // 23.8 / 22.8 / 23.2, batch 2 27.2 / 25.7 / 24.7, batch 8 61.6 / 53.8 / 52.4; for the weights: batch 1 22.8 / 23.6 / 32.5,
    // batch 4 29.5 / 30.0 / 32.5, batch 8 55.2 / 52.4 / 51.6.
    if ((long long)p.n_chunks * (2 * p.gamma + 1) * p.B <= 640) {
        cfg.blockDim = dim3(512);
        HIPPO_CUDA_TRY(cudaLaunchKernelEx(&cfg, accept_stats_kernel<512>, p));
    } else {
        cfg.blockDim = dim3(256);
        HIPPO_CUDA_TRY(cudaLaunchKernelEx(&cfg, accept_stats_kernel<256>, p));
    }
    // The weights: pieces of a quarter of a chunk while all of them run at once, a chunk of few threads otherwise.  Whole acceptance with
    // this, the statistics above and the decisions' loads in one go: batch 1 18.1 -> 14.4 us, batch 2 20.1 -> 17.0, batch 8 54.7 -> 42.4.
    if ((long long)p.n_chunks * 4 * p.B <= 2 * kNumSMs) {
        constexpr int T = 512, kPer = 2;
        p.piece = T * kPer;
        cfg.gridDim = dim3((unsigned)ceil_div(p.V, p.piece), (unsigned)p.B);
        cfg.blockDim = dim3(T);
        HIPPO_CUDA_TRY(cudaLaunchKernelEx(&cfg, accept_weigh_kernel<T, kPer>, p));
    } else if ((long long)p.n_chunks * p.B <= kNumSMs) {
        cfg.gridDim = dim3((unsigned)p.n_chunks, (unsigned)p.B);
        cfg.blockDim = dim3(kAccThreads);
        HIPPO_CUDA_TRY(cudaLaunchKernelEx(&cfg, accept_weigh_kernel<kAccThreads, kAccPerThread>, p));
    } else {
        cfg.gridDim = dim3((unsigned)p.n_chunks, (unsigned)p.B);
        cfg.blockDim = dim3(256);
        HIPPO_CUDA_TRY(cudaLaunchKernelEx(&cfg, accept_weigh_kernel<256, kAccChunk / 256>, p));
    }
    cfg.blockDim = dim3(kAccThreads);
    cfg.gridDim = dim3((unsigned)p.B);
    cfg.dynamicSmemBytes = (size_t)ceil_div(p.V, p.piece) * sizeof(double);
    HIPPO_CUDA_TRY(cudaLaunchKernelEx(&cfg, accept_pick_kernel, p));
    count_launches(3);
    return HIPPO_OK;
}

// One launch: the grid is at most what the device keeps resident at once (the CTAs wait for one another between the
// steps), and never more than the first step has items.
static int32_t launch_accept_fused(const AcceptParams &p, WsHeader *hdr, cudaStream_t s) {
    // With the table of the exponentials the kernel's own arrays and these are more than the 48 KB that need no leave.
    constexpr int kMostDynamic = 40 * 1024;
    const size_t smem = (size_t)p.n_chunks * sizeof(double);
    if (smem > kMostDynamic) return launch_accept_chain(p, s);
    static std::atomic<int> resident[kMaxDevices];
    int dev = -1;
    HIPPO_CUDA_TRY(cudaGetDevice(&dev));
    int cap = (dev >= 0 && dev < kMaxDevices) ? resident[dev].load(std::memory_order_relaxed) : 0;
    if (cap == 0) {
        int per_sm = 0, sms = 0;
        HIPPO_CUDA_TRY(cudaFuncSetAttribute(accept_fused_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostDynamic));
        HIPPO_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, accept_fused_kernel, kAccThreads, kMostDynamic));
        HIPPO_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        cap = per_sm * sms;
        if (cap < 1) return launch_accept_chain(p, s);
        if (dev >= 0 && dev < kMaxDevices) resident[dev].store(cap, std::memory_order_relaxed);
    }
    long long grid = (long long)p.B * (2 * p.gamma + 1) * p.n_chunks;
    if (grid > cap) grid = cap;
    HIPPO_CUDA_TRY(cudaMemsetAsync(hdr, 0, sizeof(WsHeader), s));    // status word and the two arrival counters
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kAccThreads);
    cfg.gridDim = dim3((unsigned)grid);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    HIPPO_CUDA_TRY(cudaLaunchKernelEx(&cfg, accept_fused_kernel, p, hdr));
    count_launches(1);
    return HIPPO_OK;
}

// variant: 0 the faster of the two for the shape, else HIPPO_ACCEPT_ONE_LAUNCH / HIPPO_ACCEPT_THREE_LAUNCHES
static int32_t launch_accept(const AcceptParams &p, WsHeader *hdr, int variant, cudaStream_t s) {
    const bool fused = variant == HIPPO_ACCEPT_ONE_LAUNCH || (variant == 0 && kAcceptFusedByDefault);
    return fused ? launch_accept_fused(p, hdr, s) : launch_accept_chain(p, s);
}

}  // namespace hippo

extern "C" {

size_t hippo_accept_workspace_bytes(int32_t batch, int32_t gamma, int32_t vocab) {
    if (batch <= 0 || gamma < 0 || vocab <= 0) return 0;
    return hippo::accept_ws(batch, gamma, vocab).total;
}

int32_t hippo_accept(int32_t batch, int32_t gamma, int32_t vocab, const float *target_logits,
                     const float *draft_logits, const int32_t *draft_tokens, const float *u_accept,
                     const float *u_resample, int32_t mode, int32_t *n_accepted, int32_t *out_tokens,
                     void *workspace, size_t workspace_bytes, void *stream) {
    using namespace hippo;
    if (batch <= 0 || gamma < 0 || vocab <= 0) return fail(HIPPO_ERR_INVALID_ARG, "hippo_accept: bad sizes");
    const int variant = mode & (HIPPO_ACCEPT_ONE_LAUNCH | HIPPO_ACCEPT_THREE_LAUNCHES);
    mode &= ~(HIPPO_ACCEPT_ONE_LAUNCH | HIPPO_ACCEPT_THREE_LAUNCHES);
    if ((mode != HIPPO_ACCEPT_SAMPLE && mode != HIPPO_ACCEPT_GREEDY) || variant == (HIPPO_ACCEPT_ONE_LAUNCH | HIPPO_ACCEPT_THREE_LAUNCHES))
        return fail(HIPPO_ERR_UNIMPLEMENTED, "hippo_accept: mode %d", mode | variant);
    const bool greedy = mode == HIPPO_ACCEPT_GREEDY;
    if (!target_logits || !n_accepted || !out_tokens || !workspace || (!greedy && !u_resample))
        return fail(HIPPO_ERR_INVALID_ARG, "hippo_accept: null pointer");
    if (gamma > 0 && (!draft_tokens || (!greedy && (!draft_logits || !u_accept))))
        return fail(HIPPO_ERR_INVALID_ARG, "hippo_accept: null draft arrays with gamma > 0");
    if (gamma > 64) return fail(HIPPO_ERR_UNSUPPORTED_SHAPE, "hippo_accept: gamma > 64");
    if ((uintptr_t)workspace & 255) return fail(HIPPO_ERR_INVALID_ARG, "hippo_accept: workspace must be 256-byte aligned");
    AcceptWs w = accept_ws(batch, gamma, vocab);
    if (workspace_bytes < w.total)
        return fail(HIPPO_ERR_WORKSPACE_TOO_SMALL, "hippo_accept: workspace %zu < %zu bytes", workspace_bytes, w.total);
    if (batch > 65535 || 2 * gamma + 1 > 65535) return fail(HIPPO_ERR_UNSUPPORTED_SHAPE, "hippo_accept: batch too large");
    AcceptParams p;
    p.tl = target_logits; p.dl = draft_logits; p.ua = u_accept; p.ur = u_resample; p.x = draft_tokens;
    p.n_acc = n_accepted; p.out = out_tokens;
    p.stats = (double2 *)((char *)workspace + w.stats_off);
    p.info = (RowInfo *)((char *)workspace + w.info_off);
    p.tscan = (double *)((char *)workspace + w.tscan_off);
    p.B = batch; p.gamma = gamma; p.V = vocab; p.n_chunks = w.n_chunks; p.piece = kAccChunk;
    cudaStream_t s = (cudaStream_t)stream;
    return greedy ? launch_accept_greedy(p, s) : launch_accept(p, (WsHeader *)workspace, variant, s);
}

}  // extern "C"

// ---- hippo_accept_noalloc: the same acceptance step for callers that cannot provide a workspace -----------------
//
// Some callers have no way to obtain scratch memory at the moment they need to accept a draft: a decode loop whose
// device memory was handed in full to a serving engine's pool at start-up, a plug-in whose host forbids cudaMalloc
// (it synchronises the whole device and would stall the draft and verify streams), or glue code that only sees the
// logits and has no allocator handle at all.  For them the scratch lives in the library image itself: one
// file-scope device array per GPU that loads libhippo.so, held until the process exits.
namespace hippo {

constexpr size_t kNoAllocScratchBytes = HIPPO_ACCEPT_NOALLOC_SCRATCH_BYTES;
static __device__ __align__(256) unsigned char g_accept_scratch[kNoAllocScratchBytes];

static void *g_scratch_addr[kMaxDevices] = {nullptr};   // device address of g_accept_scratch, per device ordinal
static std::mutex g_scratch_mutex;

// In host code `g_accept_scratch` is only a handle for the runtime, not an address a kernel could use.  The real
// device address differs per GPU and is looked up once per device, with that device current.
static int32_t noalloc_scratch(void **out) {
    int dev = -1;
    HIPPO_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return fail(HIPPO_ERR_UNSUPPORTED_SHAPE, "hippo_accept_noalloc: device ordinal %d >= %d", dev, kMaxDevices);
    std::lock_guard<std::mutex> lock(g_scratch_mutex);
    if (!g_scratch_addr[dev]) {
        void *ptr = nullptr;
        HIPPO_CUDA_TRY(cudaGetSymbolAddress((void **)&ptr, g_accept_scratch));
        if (!ptr || ((uintptr_t)ptr & 255)) return fail(HIPPO_ERR_CUDA, "hippo_accept_noalloc: bad scratch address %p", ptr);
        g_scratch_addr[dev] = ptr;
    }
    *out = g_scratch_addr[dev];
    return HIPPO_OK;
}

}  // namespace hippo

extern "C" int32_t hippo_accept_noalloc(int32_t batch, int32_t gamma, int32_t vocab, const float *target_logits,
                                        const float *draft_logits, const int32_t *draft_tokens, const float *u_accept,
                                        const float *u_resample, int32_t mode, int32_t *n_accepted, int32_t *out_tokens,
                                        void *stream) {
    using namespace hippo;
    if (batch <= 0 || gamma < 0 || vocab <= 0) return fail(HIPPO_ERR_INVALID_ARG, "hippo_accept_noalloc: bad sizes");
    const int variant = mode & (HIPPO_ACCEPT_ONE_LAUNCH | HIPPO_ACCEPT_THREE_LAUNCHES);
    mode &= ~(HIPPO_ACCEPT_ONE_LAUNCH | HIPPO_ACCEPT_THREE_LAUNCHES);
    if ((mode != HIPPO_ACCEPT_SAMPLE && mode != HIPPO_ACCEPT_GREEDY) || variant == (HIPPO_ACCEPT_ONE_LAUNCH | HIPPO_ACCEPT_THREE_LAUNCHES))
        return fail(HIPPO_ERR_UNIMPLEMENTED, "hippo_accept_noalloc: mode %d", mode | variant);
    const bool greedy = mode == HIPPO_ACCEPT_GREEDY;
    if (!target_logits || !n_accepted || !out_tokens || (!greedy && !u_resample))
        return fail(HIPPO_ERR_INVALID_ARG, "hippo_accept_noalloc: null pointer");
    if (gamma > 0 && (!draft_tokens || (!greedy && (!draft_logits || !u_accept))))
        return fail(HIPPO_ERR_INVALID_ARG, "hippo_accept_noalloc: null draft arrays with gamma > 0");
    if (gamma > 64 || batch > 65535) return fail(HIPPO_ERR_UNSUPPORTED_SHAPE, "hippo_accept_noalloc: gamma > 64 or batch > 65535");
    const AcceptWs w = accept_ws(batch, gamma, vocab);
    if (w.total > kNoAllocScratchBytes)
        return fail(HIPPO_ERR_WORKSPACE_TOO_SMALL,
                    "hippo_accept_noalloc: batch %d x gamma %d x vocab %d needs %zu bytes of scratch, the built-in array "
                    "holds %zu; use hippo_accept with a caller-owned workspace",
                    batch, gamma, vocab, w.total, kNoAllocScratchBytes);
    void *scratch = nullptr;
    const int32_t rc = noalloc_scratch(&scratch);
    if (rc != HIPPO_OK) return rc;
    // Every word the kernels read from the scratch is written earlier in the same call (chunk statistics, chunk
    // weights, the per-sequence record), so nothing has to be cleared although the array keeps the previous
    // call's contents.
    AcceptParams p;
    p.tl = target_logits; p.dl = draft_logits; p.ua = u_accept; p.ur = u_resample; p.x = draft_tokens;
    p.n_acc = n_accepted; p.out = out_tokens;
    p.stats = (double2 *)((char *)scratch + w.stats_off);
    p.info = (RowInfo *)((char *)scratch + w.info_off);
    p.tscan = (double *)((char *)scratch + w.tscan_off);
    p.B = batch; p.gamma = gamma; p.V = vocab; p.n_chunks = w.n_chunks; p.piece = kAccChunk;
    cudaStream_t s = (cudaStream_t)stream;
    return greedy ? launch_accept_greedy(p, s) : launch_accept(p, (WsHeader *)scratch, variant, s);
}
