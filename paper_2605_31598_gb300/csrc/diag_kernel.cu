// App. A assumption diagnostics on the GPU.
//
//   scores_reduce       layer-level score of every key of a full-attention
//                       frame: the attention kernel's per-(KV head, query
//                       tile) partials summed in one fixed order (App. A's
//                       shared protocol sums the weights over the frame's
//                       queries within each head, then over the heads)
//   topb_mask           top-B membership of each row, ties to the lower
//                       position: an MSB-first radix select over the score
//                       bits (11 + 11 + 9), then, among scores equal to the
//                       threshold, the lowest positions
//   concentration_sums  App. A.1: mass of the top-B historical keys and of
//                       all historical keys
//   state_metrics       App. A.2: the counts and weights behind candidate-pool
//                       recall, weighted recall, retention and churn
// A few dozen rows of tens of thousands of scores are too few CTAs at one per
// row, and each CTA then walks its row alone: 28 rows of 25k scores took 42 us
// (top-B: up to eight passes), 25 us (concentration: two fp64 adds per score on
// 28 SMs) and 38 us (metrics).  A long row is therefore shared by the CTAs of one
// thread-block cluster (row_cluster), which merge their histograms and sums in
// distributed shared memory: 15, 8 and 9 us.  A row that one CTA takes alone has a
// kernel without the merging: 28 rows of 2048 in 5.2, 4.3 and 5.3 us, where a
// cluster of one took 7.9, 5.8 and 6.5.  Sums are
// added in one fixed order for a given cluster size, so they are deterministic.
#include "sm103_ptx.cuh"
#include "statekv_kernels.cuh"

namespace statekv {
namespace {

constexpr int kDiagThreads = 512;

constexpr int kDiagWarps = kDiagThreads / 32;
constexpr int kDiagBatch = 8;  // scores per thread in flight (and kept between passes)

// Sums of two doubles per thread over the block; thread 0 gets them.  An fp64
// add of a warp takes 16 cycles of the SM, so the warps reduce both values at
// once, one in each half (5 adds where two full trees take 10).  `some`: the warp has
// entries at all (a short row leaves most without: concentration of 2000 rows of 64
// 28.7 -> 20.9 us).
__device__ void block_sum2(double a, double b, bool some, double* sh, double (&out)[2])
{
    static_assert(kDiagWarps == 16, "one warp adds the warps' two sums");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool up = lane >= 16;
    double x = 0.0;
    if (some) {
        x = (up ? b : a) + __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    }
    if ((lane & 15) == 0) sh[(up ? kDiagWarps : 0) + warp] = x;
    __syncthreads();
    if (warp == 0) {
        x = sh[lane];
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        out[0] = x;
        out[1] = __shfl_sync(0xffffffffu, x, 16);
    }
    __syncthreads();
}

// Sum of one count per thread over the block (fewer than 2^32); thread 0 gets it.
__device__ unsigned block_count(unsigned x, unsigned* sh)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    x = __reduce_add_sync(0xffffffffu, x);
    if (lane == 0) sh[warp] = x;
    __syncthreads();
    if (warp == 0) x = __reduce_add_sync(0xffffffffu, lane < kDiagWarps ? sh[lane] : 0u);
    __syncthreads();
    return x;
}

// The CTA's share [lo, hi) of the row's entries [0, n): rank r of C.
__device__ __forceinline__ void row_share(long long n, int r, int C, long long& lo, long long& hi)
{
    const long long per = (n + C - 1) / C;
    lo = min(n, per * r);
    hi = min(n, lo + per);
}

__global__ void scores_reduce(const ScoresParams p)
{
    const int u = blockIdx.y;
    const long long j = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (j >= p.ncols) return;
    const int ua = p.units.unit_abs(u);
    const long long L = static_cast<long long>(p.frames[static_cast<size_t>(ua) * p.Hkv]) * p.T;
    float s = 0.f;
    if (j < L + p.T) {
        const long long col = j < L ? j : p.Bp + (j - L);
        const float* part = p.partials + static_cast<size_t>(u) * p.Hkv * p.MT * p.Pp + col;
        for (int h = 0; h < p.Hkv; ++h) {
            float sh = 0.f;  // one KV head: its query tiles in order
            for (int mt = 0; mt < p.MT; ++mt)
                sh += part[(static_cast<size_t>(h) * p.MT + mt) * p.Pp];
            s += sh;
        }
    }
    p.scores[static_cast<size_t>(u) * p.ncols + j] = s;
}

// Order-preserving bits of a (non-negative) score.  Negative scores and NaN
// count as 0.
__device__ __forceinline__ unsigned score_bits(float x)
{
    return __float_as_uint(x > 0.f ? x : 0.f);  // also maps NaN to 0
}

__device__ __forceinline__ unsigned ld_dsmem_u32(uint32_t addr)
{
    unsigned v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ double ld_dsmem_f64(uint32_t addr)
{
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void red_dsmem_add(uint32_t addr, unsigned v)
{
    asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// The cluster's partial sums, one set per CTA, added in rank order by the first (a
// CTA alone writes its own).
template <bool kCluster, int K>
__device__ void row_total(const double (&v)[K], double* sh, int r, int C, double* out)
{
    if constexpr (!kCluster) {
        if (threadIdx.x == 0)
#pragma unroll
            for (int i = 0; i < K; ++i) out[i] = v[i];
        return;
    }
    if (threadIdx.x == 0)
#pragma unroll
        for (int i = 0; i < K; ++i) sh[i] = v[i];
    ptx::cluster_sync();
    if (r == 0 && threadIdx.x < K) {
        double t = 0.0;
        for (int q = 0; q < C; ++q)
            t += ld_dsmem_f64(ptx::dsmem_addr(ptx::smem_addr(sh + threadIdx.x), q));
        out[threadIdx.x] = t;
    }
    ptx::cluster_sync();
}

constexpr int kTopbBins = 2048;

// The calls of one launch, blockIdx.y each.
constexpr int kTopbJobs = 16;
struct TopbJobs {
    struct {
        const float* scores;
        uint8_t* mask;
        long long n, B;
    } job[kTopbJobs];
};

// One cluster of C CTAs per row.  Every pass, each CTA counts its share's digits,
// adds the non-empty bins to the first CTA's counts of that pass, and finds the
// bin of the k-th largest key in the merged counts.  The result is the mask, or
// (kSums) the two sums of concentration_kernel over it, taken from the registers
// that hold the row: same order, same bits, no mask written or read.  Several
// budgets, or the two frames of the state metrics, go in one launch: 28 rows on
// eight CTAs each leave half of the thread slots idle.  Mask, concentration at two
// budgets and state metrics of 28 rows of 25k: nine launches 248 us, four 204 (what
// is left is mostly the host's: two copies of results and the calls).
template <bool kSums, bool kCluster>
__global__ void __launch_bounds__(kDiagThreads) topb_kernel(const __grid_constant__ TopbJobs jobs,
                                                            long long stride, double* out, int C)
{
    __shared__ __align__(16) unsigned hist[kTopbBins];
    __shared__ __align__(16) unsigned merged[kCluster ? 3 : 1][kCluster ? kTopbBins : 1];
    __shared__ __align__(16) unsigned eq_before[kDiagBatch * kDiagWarps];
    __shared__ unsigned wsum[kDiagWarps];
    __shared__ unsigned sh_bin, sh_count, sh_equal;
    __shared__ unsigned long long sh_k;
    const int r = kCluster ? blockIdx.x % C : 0, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long rowi = kCluster ? blockIdx.x / C : blockIdx.x;
    const long long n = jobs.job[blockIdx.y].n, B = jobs.job[blockIdx.y].B;
    const float* row = jobs.job[blockIdx.y].scores + static_cast<size_t>(rowi) * stride;
    uint8_t* mrow = kSums ? nullptr : jobs.job[blockIdx.y].mask + static_cast<size_t>(rowi) * stride;
    long long lo, hi;
    row_share(n, r, C, lo, hi);
    // this thread's entries base + tid + e kDiagThreads of a batch, as score bits
    // (kSums: as they are, for the sums)
    unsigned x[kDiagBatch] = {};
    auto bits = [](unsigned v) { return kSums ? score_bits(__uint_as_float(v)) : v; };
    auto load = [&](long long base) {
#pragma unroll
        for (int e = 0; e < kDiagBatch; ++e) {
            const long long i = base + tid + e * kDiagThreads;
            x[e] = i >= hi ? 0u : kSums ? __float_as_uint(row[i]) : score_bits(row[i]);
        }
    };
    constexpr long long kStep = kDiagBatch * kDiagThreads;
    const bool cached = hi - lo <= kStep;  // the share stays in registers
    const bool none = B <= 0, all = n <= B;
    unsigned thr = 0, tmask = 0;           // kept: (bits & tmask) > thr, or equal and among the first `ties`
    unsigned long long ties = ~0ull;       // equal entries to keep, in position order (~0: all)
    if (!none && !all) {
        if (cached) load(lo);
        if constexpr (kCluster) {
            for (int i = tid; i < 3 * kTopbBins; i += kDiagThreads) (&merged[0][0])[i] = 0;
            ptx::cluster_sync();
        }
        unsigned long long k = static_cast<unsigned long long>(B);
#pragma unroll 1
        for (int pass = 0; pass < 3; ++pass) {
            const int shift = pass == 0 ? 20 : pass == 1 ? 9 : 0;
            const unsigned dmask = pass == 2 ? 0x1FFu : 0x7FFu;
            static_assert(kTopbBins == 4 * kDiagThreads, "four bins per thread");
            *reinterpret_cast<uint4*>(hist + 4 * tid) = make_uint4(0u, 0u, 0u, 0u);
            __syncthreads();
            for (long long base = lo; base < hi; base += kStep) {
                if (!cached) load(base);
#pragma unroll
                for (int e = 0; e < kDiagBatch; ++e)
                    if (base + tid + e * kDiagThreads < hi && (bits(x[e]) & tmask) == thr)
                        atomicAdd(&hist[(bits(x[e]) >> shift) & dmask], 1u);
            }
            __syncthreads();
            // the bin, from the largest digit down: thread t owns the four digits
            // 2047 - 4 t - j (one 16-byte load: as four words, the eight CTAs'
            // remote reads of one SM took 6 us a pass)
            float4 c4;
            if constexpr (kCluster) {
                const uint32_t m0 = ptx::dsmem_addr(ptx::smem_addr(merged[pass]), 0);
                for (int i = tid; i < kTopbBins; i += kDiagThreads)
                    if (hist[i]) red_dsmem_add(m0 + 4 * i, hist[i]);
                ptx::cluster_sync();
                c4 = ptx::ld_dsmem_f4(m0 + 4 * (kTopbBins - 4 - 4 * tid));
            } else {
                c4 = *reinterpret_cast<const float4*>(hist + kTopbBins - 4 - 4 * tid);
            }
            const unsigned c[4] = {__float_as_uint(c4.w), __float_as_uint(c4.z), __float_as_uint(c4.y),
                                   __float_as_uint(c4.x)};
            const unsigned local = c[0] + c[1] + c[2] + c[3];
            unsigned incl = local;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (lane == 31) wsum[warp] = incl;
            __syncthreads();
            unsigned long long above = incl - local;
            for (int w = 0; w < warp; ++w) above += wsum[w];
            if (above < k && above + local >= k) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (above < k && above + c[j] >= k) {
                        sh_bin = kTopbBins - 1 - 4 * tid - j;
                        sh_count = c[j];
                        sh_k = k - above;
                    }
                    above += c[j];
                }
            }
            __syncthreads();
            thr |= sh_bin << shift;
            tmask |= dmask << shift;
            k = sh_k;
            if (sh_count == k) break;  // every entry of the bin is kept
            if (pass == 2) ties = k;
        }
        if constexpr (kCluster) {
            if (ties != ~0ull) {
                // the k lowest positions among the entries equal to the threshold: the
                // CTAs' counts of them, in rank order, are in their last histograms
                if (tid == 0) sh_equal = hist[thr & 0x1FFu];
                ptx::cluster_sync();
                unsigned long long before = 0;
                for (int q = 0; q < r; ++q) before += ld_dsmem_u32(ptx::dsmem_addr(ptx::smem_addr(&sh_equal), q));
                ties = before < ties ? ties - before : 0;
            }
            ptx::cluster_sync();  // no CTA leaves while others read its shared memory
        }
    }
    // kept(j) <=> j < n and key(j) above the threshold, or equal and in time
    unsigned long long seen = 0;  // equal entries of this CTA's earlier batches
    double top = 0.0, rest = 0.0;
    for (long long base = lo; base < hi; base += kStep) {
        if (none || all ? kSums : !cached) load(base);
        unsigned eq[kDiagBatch];  // lanes of the warp whose entry equals the threshold
        if (ties != ~0ull) {
            // how many come before, in position order: the warps' counts of the batch,
            // entry e of every warp before entry e + 1, added up by the first warp (three
            // barriers a batch; two for each e, 2000 rows of 64 equal scores took 83 us)
            if (base > lo) __syncthreads();  // the previous batch's have been read
#pragma unroll
            for (int e = 0; e < kDiagBatch; ++e) {
                eq[e] = __ballot_sync(0xffffffffu, base + tid + e * kDiagThreads < hi && (bits(x[e]) & tmask) == thr);
                if (lane == 0) eq_before[e * kDiagWarps + warp] = __popc(eq[e]);
            }
            __syncthreads();
            if (warp == 0) {
                static_assert(kDiagBatch * kDiagWarps == 128, "four counts per lane");
                uint4 q = *reinterpret_cast<const uint4*>(eq_before + 4 * lane);
                const unsigned own = q.x + q.y + q.z + q.w;
                unsigned incl = own;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                const unsigned b0 = incl - own;
                q = make_uint4(b0, b0 + q.x, b0 + q.x + q.y, b0 + q.x + q.y + q.z);
                *reinterpret_cast<uint4*>(eq_before + 4 * lane) = q;
                if (lane == 31) sh_count = incl;
            }
            __syncthreads();
        }
#pragma unroll
        for (int e = 0; e < kDiagBatch; ++e) {
            if (base + warp * 32 + e * kDiagThreads >= hi) break;  // nothing of the warp's
            const long long i = base + tid + e * kDiagThreads;
            const unsigned d = bits(x[e]) & tmask;
            bool keep = all || d > thr || (d == thr && ties == ~0ull);
            if (ties != ~0ull && d == thr)
                keep = seen + eq_before[e * kDiagWarps + warp] + __popc(eq[e] & ((1u << lane) - 1)) < ties;
            if constexpr (kSums) {
                const bool in = i < hi && !none && keep;
                const double t = (in ? top : rest) + __uint_as_float(x[e]);
                top = in ? t : top;
                rest = in ? rest : t;
            } else if (i < hi) {
                mrow[i] = !none && keep ? 1 : 0;
            }
        }
        if (ties != ~0ull) seen += sh_count;
    }
    if constexpr (kSums) {
        __shared__ double sh[2 * kDiagWarps], part[2];
        double v[2] = {};
        block_sum2(top, rest, lo + warp * 32 < hi, sh, v);
        v[1] += v[0];
        row_total<kCluster>(v, part, r, C, out + 2 * (blockIdx.y * static_cast<size_t>(gridDim.x / C) + rowi));
        return;
    }
    long long t0, t1;  // entries past n
    row_share(stride - n, r, C, t0, t1);
    for (long long j = n + t0 + tid; j < n + t1; j += kDiagThreads) mrow[j] = 0;
}

template <bool kCluster>
__global__ void __launch_bounds__(kDiagThreads) concentration_kernel(const float* scores,
                                                                     const uint8_t* mask,
                                                                     long long n, long long stride,
                                                                     double* out, int C)
{
    __shared__ double sh[2 * kDiagWarps], part[2];
    const int r = kCluster ? blockIdx.x % C : 0;
    const long long rowi = kCluster ? blockIdx.x / C : blockIdx.x;
    const float* row = scores + static_cast<size_t>(rowi) * stride;
    const uint8_t* mrow = mask + static_cast<size_t>(rowi) * stride;
    long long lo, hi;
    row_share(n, r, C, lo, hi);
    double top = 0.0, rest = 0.0;  // one add per score: all = top + rest
    for (long long base = lo; base < hi; base += kDiagBatch * kDiagThreads) {
        float x[kDiagBatch];
        bool in[kDiagBatch];
#pragma unroll
        for (int e = 0; e < kDiagBatch; ++e) {
            const long long j = base + threadIdx.x + e * kDiagThreads;
            x[e] = j < hi ? row[j] : 0.f;
            in[e] = j < hi && mrow[j];
        }
#pragma unroll
        for (int e = 0; e < kDiagBatch; ++e) {
            if (base + (threadIdx.x & ~31u) + e * kDiagThreads >= hi) break;  // nothing of the warp's
            const double t = (in[e] ? top : rest) + x[e];
            top = in[e] ? t : top;
            rest = in[e] ? rest : t;
        }
    }
    double v[2] = {};
    block_sum2(top, rest, lo + (threadIdx.x & ~31u) < hi, sh, v);
    v[1] += v[0];
    row_total<kCluster>(v, part, r, C, out + 2 * rowi);
}

template <bool kCluster>
__global__ void __launch_bounds__(kDiagThreads) state_metrics_kernel(
    const uint8_t* mask_n, const uint8_t* mask_n1, const float* w, long long n_seen, int T,
    long long stride, double* out, int C)
{
    __shared__ double sh[2 * kDiagWarps], part[6];
    __shared__ unsigned shi[kDiagWarps];
    const int r = kCluster ? blockIdx.x % C : 0;
    const long long rowi = kCluster ? blockIdx.x / C : blockIdx.x;
    const size_t base0 = static_cast<size_t>(rowi) * stride;
    long long lo, hi;
    row_share(n_seen + T, r, C, lo, hi);
    unsigned cnt[4] = {0, 0, 0, 0};  // |S_n1 & P|, |S_n1|, |S_n & S_n1|, |S_n| (a share has < 2^32 entries)
    double in_p = 0.0, out_p = 0.0;  // w(S_n1 & P), w(S_n1 - P)
    for (long long base = lo; base < hi; base += kDiagBatch * kDiagThreads) {
        float x[kDiagBatch];
        bool a[kDiagBatch], b[kDiagBatch], pool[kDiagBatch];
#pragma unroll
        for (int e = 0; e < kDiagBatch; ++e) {
            const long long j = base + threadIdx.x + e * kDiagThreads;
            a[e] = j < hi && j < n_seen && mask_n[base0 + j];  // in S_n
            b[e] = j < hi && mask_n1[base0 + j] != 0;          // in S_n1
            pool[e] = a[e] || j >= n_seen;                     // S_n plus frame n + 1
            x[e] = j < hi ? w[base0 + j] : 0.f;
        }
#pragma unroll
        for (int e = 0; e < kDiagBatch; ++e) {
            if (base + (threadIdx.x & ~31u) + e * kDiagThreads >= hi) break;  // nothing of the warp's
            cnt[0] += b[e] && pool[e];
            cnt[1] += b[e];
            cnt[2] += a[e] && b[e];
            cnt[3] += a[e];
            const double t = (pool[e] ? in_p : out_p) + (b[e] ? x[e] : 0.f);
            in_p = pool[e] ? t : in_p;
            out_p = pool[e] ? out_p : t;
        }
    }
    double wt[2] = {};
    block_sum2(in_p, out_p, lo + (threadIdx.x & ~31u) < hi, sh, wt);
    double v[6];
    v[0] = block_count(cnt[0], shi);
    v[1] = block_count(cnt[1], shi);
    v[2] = wt[0];
    v[3] = wt[0] + wt[1];
    v[4] = block_count(cnt[2], shi);
    v[5] = block_count(cnt[3], shi);
    row_total<kCluster>(v, part, r, C, out + 6 * rowi);
}

// CTAs per row, a power of two up to 8 (the portable cluster size): doubled while the
// row's share is more than a batch (4096 entries, what a CTA's registers hold) and the
// CTAs of all rows stay one per SM (sixteen clusters of eight, two per GPC of 19 SMs), or
// three per SM while a share is more than eight batches.  Top-B of 28 rows, with equal
// scores in brackets, on 1, 2, 4 and 8 CTAs a row: 4097 entries 7.5 (8.8), 8.6 (9.6), 9.3
// (10.6), 14.0 (16.9) us; 9000 10.6 (12.5), 12.8 (14.4), 9.8 (11.1), 13.0 (16.9); 25k 24.3
// (25.3), 21.6 (22.2), 16.4 (16.8), 17.1 (18.2); sums and metrics prefer two to one from
// 4097 on (4097 13.7 and 11.7 us together).  8 rows of 25k 21.1, 19.4, 14.9, 12.6; 152 rows
// of 25k 21.3, 25.9, 34.9, 55.2; 100 rows of 80k 68.8, 55.3, 46.1, 64.1.  (Several jobs a
// launch keep the C of one, so the sums do too.  The 152 SMs are written in: a call may
// come before any handle has read the device's count, and the order of the sums should not
// follow it.)
int row_cluster(int rows, long long n)
{
    constexpr long long kBatch = kDiagBatch * kDiagThreads, kSms = 152;
    int C = 1;
    while (C < 8 && n > C * kBatch) {
        const long long ctas = 2ll * C * rows;
        if (ctas > (n > 8 * C * kBatch ? 3 * kSms : C == 4 ? 128 : kSms)) break;
        C *= 2;
    }
    return C;
}

// `clustered` on C CTAs per row, `alone` (no cluster, nothing to merge) where C is 1.
template <class... KArgs, class... Args>
cudaError_t launch_rows(void (*clustered)(KArgs...), void (*alone)(KArgs...), int rows, int jobs, int C,
                        cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(static_cast<unsigned>(rows) * C, static_cast<unsigned>(jobs));
    cfg.blockDim = dim3(kDiagThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = C > 1 ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, C > 1 ? clustered : alone, args..., C);
}

}  // namespace

cudaError_t launch_scores_reduce(const ScoresParams& p, int U, cudaStream_t st)
{
    if (U <= 0 || p.ncols <= 0) return cudaSuccess;
    const dim3 grid(static_cast<unsigned>((p.ncols + 255) / 256), static_cast<unsigned>(U));
    scores_reduce<<<grid, 256, 0, st>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_topb_mask(const float* scores, int rows, long long n, long long stride,
                             long long B, uint8_t* mask, cudaStream_t st)
{
    if (rows <= 0) return cudaSuccess;
    TopbJobs jobs{};
    jobs.job[0] = {scores, mask, n, B};
    return launch_rows(topb_kernel<false, true>, topb_kernel<false, false>, rows, 1, row_cluster(rows, n), st, jobs,
                       stride, static_cast<double*>(nullptr));
}

cudaError_t launch_topb_concentration(const float* scores, int rows, long long n, long long stride,
                                      const int64_t* budgets, int count, double* out, cudaStream_t st)
{
    if (rows <= 0) return cudaSuccess;
    for (int b0 = 0; b0 < count; b0 += kTopbJobs) {
        const int nb = count - b0 < kTopbJobs ? count - b0 : kTopbJobs;
        TopbJobs jobs{};
        for (int i = 0; i < nb; ++i) jobs.job[i] = {scores, nullptr, n, budgets[b0 + i]};
        const cudaError_t e = launch_rows(topb_kernel<true, true>, topb_kernel<true, false>, rows, nb,
                                          row_cluster(rows, n), st, jobs, stride,
                                          out + static_cast<size_t>(b0) * rows * 2);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_topb_metrics(const float* scores_n, const float* scores_n1, int rows, long long n_seen, int T,
                                long long stride, long long B, uint8_t* mask_n, uint8_t* mask_n1, double* out,
                                cudaStream_t st)
{
    if (rows <= 0) return cudaSuccess;
    TopbJobs jobs{};
    jobs.job[0] = {scores_n, mask_n, n_seen, B};
    jobs.job[1] = {scores_n1, mask_n1, n_seen + T, B};
    const cudaError_t e = launch_rows(topb_kernel<false, true>, topb_kernel<false, false>, rows, 2,
                                      row_cluster(rows, n_seen + T), st, jobs, stride, static_cast<double*>(nullptr));
    return e != cudaSuccess ? e
                            : launch_state_metrics(mask_n, mask_n1, scores_n1, rows, n_seen, T, stride, out, st);
}

cudaError_t launch_concentration(const float* scores, const uint8_t* mask, int rows, long long n,
                                 long long stride, double* out, cudaStream_t st)
{
    if (rows <= 0) return cudaSuccess;
    return launch_rows(concentration_kernel<true>, concentration_kernel<false>, rows, 1, row_cluster(rows, n), st,
                       scores, mask, n, stride, out);
}

cudaError_t launch_state_metrics(const uint8_t* mask_n, const uint8_t* mask_n1, const float* w,
                                 int rows, long long n_seen, int T, long long stride, double* out,
                                 cudaStream_t st)
{
    if (rows <= 0) return cudaSuccess;
    return launch_rows(state_metrics_kernel<true>, state_metrics_kernel<false>, rows, 1,
                       row_cluster(rows, n_seen + T), st, mask_n, mask_n1, w, n_seen, T, stride, out);
}

}  // namespace statekv
