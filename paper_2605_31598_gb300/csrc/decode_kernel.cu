// Decoding over the detailed cache (Sec. 3.2 / 3.3: decoding conditions on
// the detailed state D_N): a one-pass split-K attention for a few new tokens.
//
// Each of the n new tokens' G query heads of a KV head (R = n G <= 16 rows)
// attends to every cache row and, causally, to the new tokens themselves.
// Unlike the prefill kernel (two passes, so that the importance can use the
// final log-sum-exp), decoding needs no importance: one pass with an online
// max / sum per row streams each K and V row once.  The work is HBM-bound:
// at most 16 query rows meet each key, so the warp-level m16n8k16 MMA (rows
// padded to 16) keeps the instruction count far below the memory time.
//
// One launch per call, grid (chunks, KV heads, units), 4 warps:
//   append   the CTA whose key range holds the new tokens' rows writes their
//            K/V into the cache;
//   partial  a warp takes 32 keys at a time: their K and V rows arrive as TMA
//            tensor copies (boxes of 64 columns x 32 keys of the cache's 4-D
//            map, 128-byte swizzle), two steps ahead, into the warp's
//            three-stage ring, each stage behind an mbarrier; ldmatrix undoes
//            the swizzle.  Then S = Q K^T, the running max / sum per row, P in
//            bf16, O += P V.  The 4 warps' (max, sum, O) merge into the
//            chunk's partial;
//   combine  the last CTA of a (unit, KV head) to finish (a ticket per head
//            that wraps back to 0) merges the chunks' partials, rescaled to
//            the overall max and added in chunk order, into O / sum, and
//            advances the head's token count.
// A call for one layer (as a decoder makes them) moves few bytes -- 25.7 MB at
// four KV heads and 12.5k rows, 3.8 us of HBM time -- so what bounds it is the
// chain of latencies.  As four launches (append, partial, a combine of one
// thread per output element and chunk-serial loads, counter) it took 51 us per
// layer, 38 of them in the combine; this one takes 12.7 (13.5 before the keys were
// requested into L2 ahead of the previous layer's end; 5.3 of these were the
// copies, 4 the merge across CTAs).
// Every wait is bounded by the watchdog.
#include "sm103_ptx.cuh"
#include "statekv_kernels.cuh"

namespace statekv {
namespace {

using namespace ptx;

constexpr int kDecThreads = 128;
constexpr int kDecWarps = kDecThreads / 32;
constexpr int kDecKeys = kDecodeKeyBox;  // keys per warp step (one TMA box)
constexpr int kDecStages = 3; // steps a warp has in flight or in use

template <int D>
struct DecLayout {
    // a 32-key tile of K (or V): D / 64 blocks of 32 rows x 128 bytes (64
    // columns), each in the TMA's 128-byte swizzle (1 KB atoms of 8 rows)
    static constexpr int kBlock = kDecKeys * 128;
    static constexpr int kMat = (D / 64) * kBlock;
    static constexpr int kStage = 2 * kMat;                  // K and V
    static constexpr int kWarp = kDecStages * kStage;
    static constexpr int kOffBar = kDecWarps * kWarp;        // full[warp][stage]
    static constexpr int kBytes = kOffBar + kDecWarps * kDecStages * 8 + 8;  // .. landed
    static constexpr int kAlloc = kBytes + 1024;             // room to align the base to 1 KB
    static_assert(kDecWarps * kDecodeRows * (D + 8) * 4 + 2 * kDecWarps * kDecodeRows * 4 <= kOffBar &&
                      kDecodeRows * (kDecodeMaxChunks + 1) * 4 + kDecodeRows * D * 4 <= kOffBar,
                  "merge areas fit");
    // chunks whose partials of 16 rows fit the staging memory at once (23 at D = 128)
    static_assert((kOffBar - kDecodeRows * (kDecodeMaxChunks + 1) * 4) / (kDecodeRows * D * 4) >= 22,
                  "merge of every chunk in three rounds at most");
    static_assert(kBlock % 1024 == 0, "swizzle atoms stay aligned");
};

// Byte offset of element (row, col) of a swizzled 32-key tile.
__device__ __forceinline__ uint32_t sw_off(int row, int col)
{
    const int blk = col >> 6, cc = col & 63;
    return blk * (kDecKeys * 128) + row * 128 + ((((cc >> 3) ^ (row & 7))) << 4) + ((cc & 7) << 1);
}

__device__ __forceinline__ unsigned long long dec_timer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ bool dec_wait(uint64_t* bar, uint32_t parity, unsigned long long deadline)
{
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 64; ++i)
            if (mbar_try_wait(bar, parity)) return true;
        if (dec_timer() > deadline) return false;
    }
}

__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// D (16x8, fp32) += A (16x16 bf16, row) * B (16x8 bf16, col)
__device__ __forceinline__ void mma16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                         uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7},"
        " {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// four 8x8 bf16 matrices, lane l giving the 16-byte row address of row l % 8 of
// matrix l / 8; plain, or each transposed
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}

template <int D>
__global__ void __launch_bounds__(kDecThreads)
    decode_attend(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                   const DecodeParams p)
{
    using L = DecLayout<D>;
    extern __shared__ uint8_t dsm_raw[];
    uint8_t* dsm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dsm_raw) + 1023) &
                                              ~static_cast<uintptr_t>(1023));
    __shared__ int last_cta;
    const int chunk = blockIdx.x, hkv = blockIdx.y, u = blockIdx.z;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, tig = lane & 3;  // fragment row group and column pair
    const int ua = p.units.unit_abs(u);
    const size_t head = static_cast<size_t>(ua) * p.Hkv + hkv;
    uint8_t* wsm = dsm + warp * L::kWarp;
    uint64_t* full = reinterpret_cast<uint64_t*>(dsm + L::kOffBar) + warp * kDecStages;
    if (lane == 0) {
        for (int s2 = 0; s2 < kDecStages; ++s2) mbar_init(&full[s2], 1);
        if (warp == 0) mbar_init(full + kDecWarps * kDecStages, 1);  // landed, below
        fence_mbar_init();
        if (warp == 0) {
            tma_prefetch_desc(&tm_k);
            tma_prefetch_desc(&tm_v);
        }
    }
    __syncwarp();
    // The CTA's keys are requested into L2 while the stream's previous kernel ends
    // (a decoder's layers follow one another: most SMs idle while the last CTAs of the
    // previous layer merge their chunks).  The counters may be about to change, and
    // rows about to be written: this is a hint within the cache, and L2 is where
    // later writes land and the copies below read.  A lane takes 32 keys of K and V.
    if (p.prefetch) {
        const int hint = min(static_cast<long long>(__ldcg(p.frames + head)) * p.T + __ldcg(p.text + head), p.cap);
        for (int k = chunk * p.ck + 32 * static_cast<int>(threadIdx.x); k < min(hint, (chunk + 1) * p.ck);
             k += 32 * kDecThreads) {
            const uint32_t bytes = min(32, min(hint, (chunk + 1) * p.ck) - k) * D * 2;
            prefetch_l2(p.cache_k + (head * p.cap + k) * D, bytes);
            prefetch_l2(p.cache_v + (head * p.cap + k) * D, bytes);
        }
    }
    // everything above overlaps the end of the stream's previous kernel
    // (programmatic launch); nothing it wrote is used before this wait
    pdl_wait();
    pdl_launch_dependents();
    const int len0 = p.frames[head] * p.T + p.text[head];  // rows before the new tokens
    const int len = len0 + p.n;
    const int R = p.n * p.G;
    const int k0 = chunk * p.ck, k1 = min(len, k0 + p.ck);  // k1 < k0: nothing to do
    const unsigned long long deadline = dec_timer() + p.watchdog_ns;
    bool ok = true;

    // the 32 K and V rows from key `base` into stage st, by one lane (rows past
    // the cache capacity read as zero; their scores are masked)
    auto load_step = [&](int base, int st) {
        if (lane == 0) {
            uint8_t* ks = wsm + st * L::kStage;
            uint8_t* vs = ks + L::kMat;
            fence_proxy_async_smem();  // the warp's earlier reads of this stage come first
            mbar_arrive_expect_tx(&full[st], 2 * L::kMat);
#pragma unroll
            for (int hb = 0; hb < D / 64; ++hb) {
                tma_load_4d(ks + hb * L::kBlock, &tm_k, &full[st], hb * 64, base, hkv, ua);
                tma_load_4d(vs + hb * L::kBlock, &tm_v, &full[st], hb * 64, base, hkv, ua);
            }
        }
    };
    const int stride = kDecWarps * kDecKeys;
    const int base0 = k0 + warp * kDecKeys;
    const int nsteps = base0 < k1 ? (k1 - base0 + stride - 1) / stride : 0;
    // kDecStages - 1 steps ahead
#pragma unroll
    for (int s0 = 0; s0 < kDecStages - 1; ++s0)
        if (s0 < nsteps) load_step(base0 + s0 * stride, s0);
    // the new tokens' K/V rows among this CTA's keys go into the cache; nothing in
    // this launch reads them from there (put_new below), so that comes last
    const int per = D / 8;  // 16-byte chunks per row
    auto append = [&]() {
        const int r0 = max(k0, len0);
        for (int i = threadIdx.x; i < (k1 - r0) * per * 2; i += kDecThreads) {
            const int which = i / ((k1 - r0) * per), rr = i - which * (k1 - r0) * per;
            const int row = r0 + rr / per, ch = rr % per;
            if (!SKV_CHECK(row >= 0 && row < p.cap, p.status, 5)) continue;
            const size_t src = ((static_cast<size_t>(u) * p.n + (row - len0)) * p.Hkv + hkv) * D + ch * 8;
            *reinterpret_cast<uint4*>((which ? p.cache_v : p.cache_k) + (head * p.cap + row) * D + ch * 8) =
                *reinterpret_cast<const uint4*>((which ? p.v : p.k) + src);
        }
    };
    // A step that reaches the new tokens: its TMA copy brought whatever the cache
    // held there, so the warp puts their rows over it from the inputs.  (Reading
    // them back through the cache needs the writes ordered before the copy by a
    // proxy fence, which held up this CTA, and with it the head, by 1.2 us; so did
    // the append itself ahead of the loop.)
    auto put_new = [&](int base, uint8_t* ks) {
        const int lo = max(base, len0), hi = min(base + kDecKeys, k1);
        for (int i = lane; i < (hi - lo) * per * 2; i += 32) {
            const int which = i / ((hi - lo) * per), rr = i - which * (hi - lo) * per;
            const int row = lo + rr / per, ch = rr % per;
            const size_t src = ((static_cast<size_t>(u) * p.n + (row - len0)) * p.Hkv + hkv) * D + ch * 8;
            *reinterpret_cast<uint4*>(ks + which * L::kMat + sw_off(row - base, ch * 8)) =
                *reinterpret_cast<const uint4*>((which ? p.v : p.k) + src);
        }
        __syncwarp();
    };

    // Q as A fragments, while the first steps are on their way: row r = token
    // r / G, head hkv G + r % G (rows >= R are 0)
    uint32_t qa[D / 16][4];
    {
        const uint32_t* qrow[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = g + 8 * h, t = r / p.G, gg = r - t * p.G;
            qrow[h] = r < R ? reinterpret_cast<const uint32_t*>(
                                  p.q + ((static_cast<size_t>(u) * p.n + t) * p.Hq + hkv * p.G + gg) * D) + tig
                            : nullptr;
        }
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks)
#pragma unroll
            for (int e = 0; e < 4; ++e)  // e & 1: row half, e >> 1: column half
                qa[ks][e] = qrow[e & 1] ? qrow[e & 1][ks * 8 + (e >> 1) * 4] : 0u;
    }

    const float c = p.scale_log2;
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};  // rows g and g + 8
    float o[D / 8][4];
#pragma unroll
    for (int nd = 0; nd < D / 8; ++nd)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[nd][e] = 0.f;

    // ldmatrix row addresses of this lane: K matrices (8 keys) x (4 x 8 columns), V
    // matrices (2 x 8 keys) x (2 x 8 columns)
    const int lrow = lane & 7, lmat = lane >> 3;
    int step = 0;
    for (; step < nsteps; ++step) {
        const int base = base0 + step * stride;
        const int st = step % kDecStages;
        const int pre = step + kDecStages - 1;
        // the stage `pre` lands in was read by step - 1, which this warp finished
        if (pre < nsteps) load_step(base0 + pre * stride, pre % kDecStages);
        ok = __all_sync(0xffffffffu, dec_wait(&full[st], (step / kDecStages) & 1, deadline));
        if (!ok) break;
        if (base + kDecKeys > len0) put_new(base, wsm + st * L::kStage);
        const uint32_t ks = smem_addr(wsm + st * L::kStage);
        const uint32_t vs = ks + L::kMat;
        // S = Q K^T: 4 key tiles of 8
        float sc[4][4];
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
#pragma unroll
            for (int e = 0; e < 4; ++e) sc[nt][e] = 0.f;
#pragma unroll
            for (int kst = 0; kst < D / 16; kst += 2) {
                uint32_t b[4];
                ldsm4(b, ks + sw_off(nt * 8 + lrow, kst * 16 + lmat * 8));
                mma16816(sc[nt], qa[kst], b[0], b[1]);
                mma16816(sc[nt], qa[kst + 1], b[2], b[3]);
            }
        }
        // masks, running max / sum of rows g (h = 0) and g + 8 (h = 1)
        float alpha[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = g + 8 * h;
            const int lim = r < R ? min(k1, len0 + r / p.G + 1) : 0;  // keys [.., lim) visible
            float mx = -INFINITY;
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int key = base + nt * 8 + 2 * tig + e;
                    float& v = sc[nt][2 * h + e];
                    v = key < lim ? v * c : -INFINITY;
                    mx = fmaxf(mx, v);
                }
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
            const float mn = fmaxf(m[h], mx);
            alpha[h] = mn == -INFINITY ? 1.f : ex2(m[h] - mn);
            float sum = 0.f;
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    float& v = sc[nt][2 * h + e];
                    v = mn == -INFINITY ? 0.f : ex2(v - mn);
                    sum += v;
                }
            sum += __shfl_xor_sync(0xffffffffu, sum, 1);
            sum += __shfl_xor_sync(0xffffffffu, sum, 2);
            l[h] = l[h] * alpha[h] + sum;
            m[h] = mn;
        }
#pragma unroll
        for (int nd = 0; nd < D / 8; ++nd) {
            o[nd][0] *= alpha[0];
            o[nd][1] *= alpha[0];
            o[nd][2] *= alpha[1];
            o[nd][3] *= alpha[1];
        }
        // O += P V: P as A fragments (keys 16j .. 16j + 15 are tiles 2j, 2j + 1)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const uint32_t pa[4] = {pack_bf16(sc[2 * j][0], sc[2 * j][1]),
                                    pack_bf16(sc[2 * j][2], sc[2 * j][3]),
                                    pack_bf16(sc[2 * j + 1][0], sc[2 * j + 1][1]),
                                    pack_bf16(sc[2 * j + 1][2], sc[2 * j + 1][3])};
#pragma unroll
            for (int nd = 0; nd < D / 8; nd += 2) {
                uint32_t b[4];
                ldsm4t(b, vs + sw_off(16 * j + (lmat & 1) * 8 + lrow, (nd + (lmat >> 1)) * 8));
                mma16816(o[nd], pa, b[0], b[1]);
                mma16816(o[nd + 1], pa, b[2], b[3]);
            }
        }
        __syncwarp();  // the stage is refilled kDecStages - 1 steps later
    }
    if (!ok) {
        if (lane == 0) *reinterpret_cast<volatile int32_t*>(p.status) = DEV_TIMEOUT_DECODE;
        // let the copies already issued land before the shared memory is reused
        if (lane == 0)
            for (int s2 = step; s2 < min(nsteps, step + kDecStages); ++s2)
                dec_wait(&full[s2 % kDecStages], (s2 / kDecStages) & 1, dec_timer() + p.watchdog_ns);
    }
    __syncthreads();

    // merge the 4 warps into the chunk's partial (reusing the staging memory;
    // rows padded by 8 floats: the fragment stores of a warp hit distinct banks)
    constexpr int kLd = D + 8;
    float* mo = reinterpret_cast<float*>(dsm);                       // [warp][16][kLd]
    float* mm = mo + kDecWarps * kDecodeRows * kLd;                   // [warp][16]
    float* ml = mm + kDecWarps * kDecodeRows;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int r = g + 8 * h;
        if (tig == 0) {
            mm[warp * kDecodeRows + r] = m[h];
            ml[warp * kDecodeRows + r] = l[h];
        }
        if (r < R)
#pragma unroll
            for (int nd = 0; nd < D / 8; ++nd)
                *reinterpret_cast<float2*>(mo + (warp * kDecodeRows + r) * kLd + nd * 8 + 2 * tig) =
                    make_float2(o[nd][2 * h], o[nd][2 * h + 1]);
    }
    __syncthreads();
    const size_t pidx = (static_cast<size_t>(u) * p.Hkv + hkv) * p.nchunk + chunk;
    float* po = p.part_o + pidx * kDecodeRows * D;
    float* pml = p.part_ml + pidx * kDecodeRows * 2;
    for (int i = threadIdx.x; i < R * (D / 4); i += kDecThreads) {
        const int r = i / (D / 4), d4 = i - r * (D / 4);
        float M = -INFINITY;
#pragma unroll
        for (int w = 0; w < kDecWarps; ++w) M = fmaxf(M, mm[w * kDecodeRows + r]);
        float4 ov = make_float4(0.f, 0.f, 0.f, 0.f);
        float Lv = 0.f;
        if (M != -INFINITY) {
#pragma unroll
            for (int w = 0; w < kDecWarps; ++w) {
                const float mw = mm[w * kDecodeRows + r];
                const float f = mw == -INFINITY ? 0.f : ex2(mw - M);
                const float4 x = *reinterpret_cast<const float4*>(mo + (w * kDecodeRows + r) * kLd + d4 * 4);
                ov.x += x.x * f;
                ov.y += x.y * f;
                ov.z += x.z * f;
                ov.w += x.w * f;
                Lv += ml[w * kDecodeRows + r] * f;
            }
        }
        *reinterpret_cast<float4*>(po + r * D + d4 * 4) = ov;
        if (d4 == 0) *reinterpret_cast<float2*>(pml + 2 * r) = make_float2(M, Lv);
    }

    // the last CTA of the head to get here merges the chunks (the barrier orders
    // the CTA's stores before one thread's fence, which publishes them all)
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last_cta = atomicInc(p.tickets + head, gridDim.x - 1) == gridDim.x - 1 ? 1 : 0;
        __threadfence();
    }
    __syncthreads();
    if (!last_cta) {
        append();
        return;
    }
    // O = sum_c O_c 2^(m_c - M) / sum_c l_c 2^(m_c - M).  One SM reads every
    // chunk's rows here (118 KB at 33 chunks of 7 rows), so all of them are
    // requested at once, as bulk copies into the idle staging memory (loads into
    // registers, 32 x 16 bytes in flight per thread, took 4.2 us, this 2.1), and
    // the factors 2^(m_c - M) and the sums are formed meanwhile, a warp per row.
    float* fac = reinterpret_cast<float*>(dsm);                 // [16][kDecodeMaxChunks]
    float* den = fac + kDecodeRows * kDecodeMaxChunks;          // [16]
    float* rows = den + kDecodeRows;                            // [chunks of a round][R][D]
    uint64_t* landed = reinterpret_cast<uint64_t*>(dsm + L::kOffBar) + kDecWarps * kDecStages;
    const int nc = p.nchunk, items = R * (D / 4);
    const int round = (L::kOffBar - kDecodeRows * (kDecodeMaxChunks + 1) * 4) / (R * D * 4);  // >= 22 chunks
    const size_t hbase = (static_cast<size_t>(u) * p.Hkv + hkv) * nc;
    auto fetch = [&](int c0) {  // warp 0: chunks [c0, c0 + round) into `rows`
        const int cnt = min(round, nc - c0);
        if (lane == 0) mbar_arrive_expect_tx(landed, cnt * R * D * 4);
        __syncwarp();
        asm volatile("fence.proxy.async;" ::: "memory");  // after this CTA's accesses and the others' stores
        for (int ch = lane; ch < cnt; ch += 32)
            bulk_load(rows + static_cast<size_t>(ch) * R * D,
                      p.part_o + (hbase + c0 + ch) * kDecodeRows * D, R * D * 4, landed);
    };
    if (warp == 0) fetch(0);
    append();
    {
        constexpr int kRows = kDecodeRows / kDecWarps, kPer = kDecodeMaxChunks / 32;
        float2 x[kRows][kPer];  // (max, sum) of the warp's rows: every load in flight at once
#pragma unroll
        for (int k = 0; k < kRows; ++k)
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                const int r = warp + k * kDecWarps, ch = lane + 32 * i;
                x[k][i] = r < R && ch < nc ? __ldcg(reinterpret_cast<const float2*>(
                                                 p.part_ml + ((hbase + ch) * kDecodeRows + r) * 2))
                                           : make_float2(-INFINITY, 0.f);
            }
#pragma unroll
        for (int k = 0; k < kRows; ++k) {
            const int r = warp + k * kDecWarps;
            if (r >= R) break;
            float M = -INFINITY, sum = 0.f;
#pragma unroll
            for (int i = 0; i < kPer; ++i) M = fmaxf(M, x[k][i].x);
#pragma unroll
            for (int o2 = 16; o2 > 0; o2 >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o2));
#pragma unroll
            for (int i = 0; i < kPer; ++i) {
                const float f = x[k][i].x == -INFINITY ? 0.f : ex2(x[k][i].x - M);
                fac[r * kDecodeMaxChunks + lane + 32 * i] = f;
                sum += x[k][i].y * f;
            }
#pragma unroll
            for (int o2 = 16; o2 > 0; o2 >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o2);
            if (lane == 0) den[r] = sum;
        }
    }
    constexpr int kItems = kDecodeRows * (D / 4) / kDecThreads;  // four-column groups per thread, at most
    float4 acc[kItems];
#pragma unroll
    for (int j = 0; j < kItems; ++j) acc[j] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int c0 = 0, ph = 0; c0 < nc; c0 += round, ph ^= 1) {
        if (c0 > 0) {
            __syncthreads();  // the previous round has been read
            if (warp == 0) fetch(c0);
        }
        if (!dec_wait(landed, ph, dec_timer() + p.watchdog_ns) && lane == 0)
            *reinterpret_cast<volatile int32_t*>(p.status) = DEV_TIMEOUT_DECODE;
        __syncthreads();  // the factors too
        const int cnt = min(round, nc - c0);
#pragma unroll
        for (int j = 0; j < kItems; ++j) {
            const int i = threadIdx.x + j * kDecThreads;
            if (i >= items) break;
            const float* f = fac + (i / (D / 4)) * kDecodeMaxChunks + c0;
            const float4* src = reinterpret_cast<const float4*>(rows) + i;
#pragma unroll 8
            for (int ch = 0; ch < cnt; ++ch) {
                const float4 x = src[ch * items];
                acc[j].x += x.x * f[ch];
                acc[j].y += x.y * f[ch];
                acc[j].z += x.z * f[ch];
                acc[j].w += x.w * f[ch];
            }
        }
    }
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
        const int i = threadIdx.x + j * kDecThreads, r = i / (D / 4), d4 = i - r * (D / 4);
        if (i >= items) break;
        const float sum = den[r];
        const int t = r / p.G, gg = r - t * p.G;
        *reinterpret_cast<uint2*>(p.out + ((static_cast<size_t>(u) * p.n + t) * p.Hq + hkv * p.G + gg) * D + d4 * 4) =
            make_uint2(pack_bf16(acc[j].x / sum, acc[j].y / sum), pack_bf16(acc[j].z / sum, acc[j].w / sum));
    }
    // every CTA of the head has read the counters
    if (threadIdx.x == 0) p.text[head] += p.n;
}

}  // namespace

cudaError_t launch_decode(const CUtensorMap& tm_k, const CUtensorMap& tm_v, const DecodeParams& p, int D,
                          int U, cudaStream_t st)
{
    if (U <= 0) return cudaSuccess;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(p.nchunk, p.Hkv, U);
    cfg.blockDim = dim3(kDecThreads);
    cfg.dynamicSmemBytes = D == 64 ? DecLayout<64>::kAlloc : DecLayout<128>::kAlloc;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return D == 64 ? cudaLaunchKernelEx(&cfg, decode_attend<64>, tm_k, tm_v, p)
                   : cudaLaunchKernelEx(&cfg, decode_attend<128>, tm_k, tm_v, p);
}

cudaError_t decode_prepare()
{
    cudaError_t e = cudaFuncSetAttribute(decode_attend<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         DecLayout<64>::kAlloc);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(decode_attend<128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                DecLayout<128>::kAlloc);
}

}  // namespace statekv
