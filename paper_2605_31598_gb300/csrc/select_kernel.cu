// K3: importance reduction, top-B state selection and evict/admit gather
//     (Sec. 3.3, Eq. 6; per layer and KV head as in App. A).
// K4: decode-cache append (Sec. 3.2 detailed state; Sec. 3.3 "append").
//
// K3 runs one CTA per (unit, KV head) (a cluster for the sums of large pools, see
// select_split), and in the same launch, after these, a few CTAs per unit
// that append the frame's K and V to the decode cache (K4's work).  It is launched
// programmatically behind the attention kernel, so it is in place when that ends.
// The append CTAs wait for that too, although they need nothing of the attention
// kernel's: what was written before it (K, V, the frame counters) is visible to this
// grid only after the wait.  Last in the grid they take no SM from a head's CTA
// (first in it, the wait cost 4 us of 227 at 28 layers; last, none).  (As a launch of
// its own on a side stream the append needed two events per frame and kept the other
// two kernels from overlapping.  Per frame, before and after: toy 17.2 and 12.1 us,
// one 7B layer 32.5 and 27.7, four small-backbone layers 34.6 and 25.6.)
//   1. importance of every pool member = the fixed-order sum of the attention
//      kernel's per-query-tile partials (deterministic); with layer-level
//      selection (App. A) the ranking score is the same sum taken over every
//      KV head of the unit, in one fixed order, so all the unit's CTAs rank
//      identically and their states keep the same positions;
//   2. if the pool (count + T) fits in B, every frame token is admitted;
//      otherwise the B best members by (score desc, position asc) are found
//      with an MSB-first radix select over the 64-bit key
//      (score bits << 32 | ~position) -- scores are non-negative floats, whose
//      bit patterns order like the values, and positions are unique, so the
//      keys are distinct and exactly B members are kept.  Digits of 11 bits from
//      the highest bit in which two keys differ leave a few dozen candidates after
//      one pass as a rule; up to kDirect of them are then ranked by counting.
//      (8-bit digits and passes to the end took three to six passes of 1.2 us, of
//      4.5 us at a pool of 16.6k: a frame with that state 107 -> 89 us);
//   3. evicted / empty slots (ascending) receive the admitted frame tokens
//      (ascending) as 128-bit row copies, and their positions are updated.
#include "append_plan.h"
#include "sm103_ptx.cuh"
#include "statekv_kernels.cuh"

#include <algorithm>

namespace statekv {
namespace {

constexpr int kSelWarps = kSelThreads / 32;
static_assert(kSelWarps <= 32, "one warp combines the warps' values");

// Exclusive block-wide scan of one int per thread; returns the total.
__device__ __forceinline__ int block_exclusive_scan(int x, int* warp_sums, int& excl)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int w = lane < kSelWarps ? warp_sums[lane] : 0;
        int wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < kSelWarps) warp_sums[lane] = wi - w;  // exclusive warp offsets
        if (lane == kSelWarps - 1) warp_sums[kSelWarps] = wi;
    }
    __syncthreads();
    excl = warp_sums[warp] + incl - x;
    return warp_sums[kSelWarps];  // warp_sums is not written again before the caller's next barrier
}

// For each of M pool members (columns col[e], active act[e]): the sum of
// x[mt * stride + col] over mt < MT, added in mt order.  K tiles' loads of all
// members (24 or 32 independent loads) are in flight before any addition.
// (Plain loads: the kernel is resident while the attention kernel still writes
// the partials, so the read-only path, which may move a load ahead of the wait, is
// not for them.)
template <int M, int K>
__device__ __forceinline__ void tiles_sum(const float* x, int MT, int stride, const int (&col)[M],
                                          const bool (&act)[M], float (&s)[M])
{
#pragma unroll
    for (int e = 0; e < M; ++e) s[e] = 0.f;
#pragma unroll 1
    for (int mt = 0; mt < MT; mt += K) {
        float v[K][M];
#pragma unroll
        for (int m = 0; m < K; ++m)
#pragma unroll
            for (int e = 0; e < M; ++e)
                v[m][e] = (act[e] && mt + m < MT) ? x[static_cast<size_t>(mt + m) * stride + col[e]] : 0.f;
#pragma unroll
        for (int m = 0; m < K; ++m)
#pragma unroll
            for (int e = 0; e < M; ++e)
                if (mt + m < MT) s[e] += v[m][e];
    }
}

// Members per thread and round where one CTA takes the pool member by member: two
// with twelve query tiles' loads in flight; or eight with four, if there are no more
// tiles than that, layer-level scores (heads to add up, a round of latencies each)
// and three or more rounds by twos.  Two layers of 32 heads, two tiles, layer-level:
// pool 4355 168 us a frame by twos, 110 by eights (133 was eights for every pool on
// the 8-bit selection); 12 layers of 12 heads, pool 1257 56 and 66 us.
constexpr int kMem = 2, kMemFewTiles = 8;
int select_members(const SelectParams& p)
{
    return (p.P & 3) != 0 && p.MT <= 4 && p.shared && p.P > 2 * kMem * kSelThreads ? kMemFewTiles : kMem;
}

// For 4 adjacent columns c0..c0+3 (16-byte aligned): the sums of
// x[mt * stride + c] over mt < MT, added in mt order, with up to 12 rows'
// 16-byte loads in flight at once (one round of L2 latency for up to 12
// query tiles).
__device__ __forceinline__ float4 rows_sum4(const float* x, int MT, int stride, int c0)
{
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (int mt = 0; mt < MT; mt += 12) {
        float4 v[12];
#pragma unroll
        for (int m = 0; m < 12; ++m)
            v[m] = mt + m < MT ? *reinterpret_cast<const float4*>(x + static_cast<size_t>(mt + m) * stride + c0)
                               : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int m = 0; m < 12; ++m)
            if (mt + m < MT) {
                s.x += v[m].x;
                s.y += v[m].y;
                s.z += v[m].z;
                s.w += v[m].w;
            }
    }
    return s;
}

// One append CTA: its share of the unit's K, then V rows, kAppendBatch copies per
// thread in flight.
template <class I>
__device__ __forceinline__ void append_share(const SelectParams& p, int u, int part)
{
    const int chunks = p.D / 8;
    const long long copies = append_copies(p.T, p.Hkv, p.D);
    const I per = static_cast<I>(copies);
    const size_t base = static_cast<size_t>(p.units.unit_abs(u)) * p.Hkv;
    const long long row0 = static_cast<long long>(p.frames[base]) * p.T;
    const uint4* k = reinterpret_cast<const uint4*>(p.k) + u * copies;
    const uint4* v = reinterpret_cast<const uint4*>(p.v) + u * copies;
    for (I i0 = part * kAppendBatch * kSelThreads + threadIdx.x; i0 < 2 * per;
         i0 += p.appenders * kAppendBatch * kSelThreads) {
        uint4 x[kAppendBatch];
#pragma unroll
        for (int e = 0; e < kAppendBatch; ++e) {
            const I i = i0 + e * kSelThreads;
            if (i < 2 * per) x[e] = i < per ? k[i] : v[i - per];
        }
#pragma unroll
        for (int e = 0; e < kAppendBatch; ++e) {
            const I i = i0 + e * kSelThreads;
            if (i >= 2 * per) break;
            const AppendAt at = append_at(i, per, p.Hkv, chunks);
            const long long row = row0 + at.t;
            if (!SKV_CHECK(row >= 0 && row < p.cap, p.status, 4)) continue;
            reinterpret_cast<uint4*>(i < per ? p.cache_k : p.cache_v)[((base + at.hkv) * p.cap + row) * chunks + at.ch] = x[e];
        }
    }
}

// The unit's CTAs (one per KV head and the append CTAs) read its frame counters;
// the last of them to finish advances them.
__device__ __forceinline__ void finish_unit(const SelectParams& p, int u, int nf)
{
    __shared__ int last;
    const size_t base = static_cast<size_t>(p.units.unit_abs(u)) * p.Hkv;
    const unsigned total = p.Hkv + p.appenders;
    __syncthreads();  // every thread has read them
    if (threadIdx.x == 0) last = atomicInc(p.tickets + base, total - 1) == total - 1 ? 1 : 0;
    __syncthreads();
    if (last)
        for (int h = threadIdx.x; h < p.Hkv; h += kSelThreads) p.frames[base + h] = nf + 1;
}

constexpr int kMaxSelSplit = 8;
constexpr int kBins = 2048;   // radix digits of 11 bits
constexpr int kDirect = 256;  // candidates ranked by counting instead of another pass
static_assert(kBins / 4 <= kSelThreads && kBins % 128 == 0, "four bins per thread, whole warps");

// kSplit: a cluster of p.split CTAs makes the keys of a head, each from its share of
// the pool's columns; they meet in the first CTA's shared memory, which goes on alone.
// kMembers: see select_members; Index: the append's, see append_narrow.  They are
// instantiations of their own: as branches of one kernel, never taken, the eight-member
// sums cost the other forms 2 to 5%, and the 64-bit append 0.6 us of a toy frame's 12.1
// and 1.1 of the 27.7 of one 7B layer.
template <bool kSplit, int kMembers, class Index>
__global__ void __launch_bounds__(kSelThreads)
    state_select_gather(const SelectParams p)
{
    constexpr int kTiles = kMembers == kMem ? 12 : 4;  // query tiles whose loads are in flight
    extern __shared__ __align__(16) uint8_t smem_raw[];
    // A kernel launched programmatically behind this one (the transformer
    // block's output projection) may start now: it requests its first weight
    // tiles, which nothing here writes, and waits for this grid's completion
    // before it reads anything else.
    ptx::pdl_launch_dependents();
    const int C = kSplit ? p.split : 1;
    const int app = static_cast<int>(blockIdx.x) - p.U * p.Hkv * C;  // append CTA, after the heads'
    if (app >= 0) {
        ptx::pdl_wait();  // K, V and the counters, written before the attention kernel
        const int u = app / p.appenders;
        const int nf0 = p.frames[static_cast<size_t>(p.units.unit_abs(u)) * p.Hkv];
        append_share<Index>(p, u, app - u * p.appenders);
        finish_unit(p, u, nf0);
        return;
    }
    const int rank = kSplit ? static_cast<int>(ptx::cluster_ctarank()) : 0;
    if (kSplit) ptx::cluster_sync();  // the cluster's CTAs run: their shared memory can be written
    ptx::pdl_wait();  // the attention kernel's partials; it has read the state
    const int T = p.T, B = p.B, P = p.P, D = p.D;
    uint64_t* key = reinterpret_cast<uint64_t*>(smem_raw);            // [P]
    uint8_t* lists = smem_raw + (static_cast<size_t>(P) * 8 + 15) / 16 * 16;
    int* free_slot = reinterpret_cast<int*>(lists);                    // [T]
    int* adm_tok = free_slot + T;                                      // [T]
    // the radix select's histogram and candidates, before the lists are made
    unsigned long long* cand = reinterpret_cast<unsigned long long*>(lists);      // [kDirect]
    unsigned* hist = reinterpret_cast<unsigned*>(lists + kDirect * 8);            // [kBins]
    __shared__ int warp_sums[kSelWarps + 1];
    __shared__ unsigned long long sh_prefix, sh_mask;
    __shared__ int sh_k, sh_in, sh_shift, sh_ncand;
    constexpr int kMaxC = kSplit ? kMaxSelSplit : 1;
    __shared__ unsigned long long warp_and[kMaxC * kSelWarps], warp_or[kMaxC * kSelWarps];

    const int unit_head = blockIdx.x / C, u = unit_head / p.Hkv, hkv = unit_head - u * p.Hkv;
    const int ua = p.units.unit_abs(u);
    const int tid = threadIdx.x, lane = tid & 31;
    const size_t head = static_cast<size_t>(ua) * p.Hkv + hkv;
    const int count = p.counts[head];
    const int nf = p.frames[head];
    const int L = nf * T;  // virtual length before this frame
    int32_t* pos = p.positions + head * B;
    const float* part = p.partials + (static_cast<size_t>(u) * p.Hkv + hkv) * p.MT * P;
    float* imp_out =
        p.importance ? p.importance + (static_cast<size_t>(u) * p.Hkv + hkv) * P : nullptr;
    const int n = count + T;
    // the counters come from the arena: a state larger than B or a negative frame
    // count would index past the pool (uniform across the CTA)
    if (!SKV_CHECK(count >= 0 && count <= B && nf >= 0, p.status, 1)) {
        if (rank == 0) finish_unit(p, u, nf);
        return;
    }
    // the cluster's CTAs take the pool a warp's worth at a time, in turn
    const int share = ((tid >> 5) * C + rank) * 32 + lane;
    auto put_key = [&](int i, uint64_t kk) {
        if (kSplit)
            ptx::st_dsmem_u64(ptx::dsmem_addr(ptx::smem_addr(key + i), 0), kk);
        else
            key[i] = kk;
    };

    // 1. importance (fixed-order sum over query tiles) and selection keys.  A
    // thread takes several pool members at once and walks the query tiles
    // outside them, so all its loads are independent (the partials come from
    // L2); each member's sum still adds the tiles in order.
    const float* part0 = p.partials + static_cast<size_t>(u) * p.Hkv * p.MT * P;
    // bits every selection key shares: the radix select starts below them
    unsigned long long kand = ~0ull, kor = 0ull;
    if (kMembers == kMem && (P & 3) == 0) {
        // Column space, four adjacent columns per thread (16-byte loads): state
        // slot c < count is member c, frame column B + t is member count + t,
        // empty slots are skipped.
        for (int g4 = share; g4 < (P >> 2); g4 += C * kSelThreads) {
            const int c0 = 4 * g4;
            int ps[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {  // positions first: their loads overlap the sums'
                // (bounded by B, not by the count, so they do not wait for the count's load)
                const int c = c0 + e;
                ps[e] = c < B ? pos[c] : 0;
            }
            const float4 s4 = rows_sum4(part, p.MT, P, c0);
            float4 r4 = s4;
            if (p.shared) {  // the ranking score: the same sums for every KV head, heads in order
                r4 = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int h2 = 0; h2 < p.Hkv; ++h2) {
                    const float4 t4 = rows_sum4(part0 + static_cast<size_t>(h2) * p.MT * P, p.MT, P, c0);
                    r4.x += t4.x;
                    r4.y += t4.y;
                    r4.z += t4.z;
                    r4.w += t4.w;
                }
            }
            const float sv[4] = {s4.x, s4.y, s4.z, s4.w}, rv[4] = {r4.x, r4.y, r4.z, r4.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int c = c0 + e;
                const int i = c < count ? c : (c >= B && c - B < T) ? count + (c - B) : -1;
                if (i < 0) continue;
                const int pe = c < count ? ps[e] : L + (c - B);
                const uint64_t kk = (static_cast<uint64_t>(__float_as_uint(rv[e])) << 32) |
                                    static_cast<uint32_t>(0xFFFFFFFFu - static_cast<uint32_t>(pe));
                put_key(i, kk);
                kand &= kk;
                kor |= kk;
                if (imp_out) imp_out[c] = sv[e];
            }
        }
    } else {  // member-wise: kMembers pool members per thread
        for (int i0 = 0; i0 < n; i0 += C * kMembers * kSelThreads) {
            int col[kMembers], ps[kMembers];
            bool act[kMembers];
            float s[kMembers], r[kMembers];
#pragma unroll
            for (int e = 0; e < kMembers; ++e) {  // positions first: their loads overlap the sums'
                const int i = i0 + share + e * C * kSelThreads;
                act[e] = i < n;
                col[e] = !act[e] ? 0 : i < count ? i : B + (i - count);
                ps[e] = !act[e] ? 0 : i < count ? pos[i] : L + (i - count);
                r[e] = 0.f;
            }
            tiles_sum<kMembers, kTiles>(part, p.MT, P, col, act, s);
            if (p.shared) {  // the ranking score: the same sums for every KV head, heads in order
                for (int h2 = 0; h2 < p.Hkv; ++h2) {
                    float sh[kMembers];
                    tiles_sum<kMembers, kTiles>(part0 + static_cast<size_t>(h2) * p.MT * P, p.MT, P, col, act, sh);
#pragma unroll
                    for (int e = 0; e < kMembers; ++e) r[e] += sh[e];
                }
            }
#pragma unroll
            for (int e = 0; e < kMembers; ++e) {
                if (!act[e]) continue;
                const int i = i0 + share + e * C * kSelThreads;
                const float rank = p.shared ? r[e] : s[e];
                const uint64_t kk = (static_cast<uint64_t>(__float_as_uint(rank)) << 32) |
                                    static_cast<uint32_t>(0xFFFFFFFFu - static_cast<uint32_t>(ps[e]));
                put_key(i, kk);
                kand &= kk;
                kor |= kk;
                if (imp_out) imp_out[col[e]] = s[e];
            }
        }
    }
    if (imp_out)
        for (int c = count + share; c < B; c += C * kSelThreads) imp_out[c] = 0.f;
    // bits in which the keys agree, a warp's at a time, at [rank][warp] of the first CTA
    if (n > B) {
        __syncwarp();
        const uint32_t ah = __reduce_and_sync(0xffffffffu, static_cast<uint32_t>(kand >> 32));
        const uint32_t al = __reduce_and_sync(0xffffffffu, static_cast<uint32_t>(kand));
        const uint32_t oh = __reduce_or_sync(0xffffffffu, static_cast<uint32_t>(kor >> 32));
        const uint32_t ol = __reduce_or_sync(0xffffffffu, static_cast<uint32_t>(kor));
        if (lane == 0) {
            const int at = rank * kSelWarps + (tid >> 5);
            const unsigned long long a = (static_cast<unsigned long long>(ah) << 32) | al;
            const unsigned long long o = (static_cast<unsigned long long>(oh) << 32) | ol;
            if (kSplit) {
                ptx::st_dsmem_u64(ptx::dsmem_addr(ptx::smem_addr(warp_and + at), 0), a);
                ptx::st_dsmem_u64(ptx::dsmem_addr(ptx::smem_addr(warp_or + at), 0), o);
            } else {
                warp_and[at] = a;
                warp_or[at] = o;
            }
        }
    }
    if (kSplit) {
        __syncwarp();
        ptx::cluster_sync();  // every key is in the first CTA's shared memory
        if (rank != 0) return;
    }
    if (B == 0) {  // no compressed state: nothing is kept
        finish_unit(p, u, nf);
        return;
    }

    // 2. top-B selection: kept(i) <=> (key[i] & mask) >= prefix
    unsigned long long prefix = 0, mask = 0;
    if (n > B) {
        // AND and OR of all keys: digits above the highest bit in which two keys
        // differ hold one value for every key, so the radix passes start at the
        // digit holding that bit
        __syncthreads();
        if (tid < 32) {  // warp 0 combines the warps' values
            unsigned long long wa = ~0ull, wo = 0ull;
            for (int i = lane; i < C * kSelWarps; i += 32) {
                wa &= warp_and[i];
                wo |= warp_or[i];
            }
            const unsigned long long a =
                (static_cast<unsigned long long>(__reduce_and_sync(0xffffffffu, static_cast<uint32_t>(wa >> 32)))
                 << 32) |
                __reduce_and_sync(0xffffffffu, static_cast<uint32_t>(wa));
            const unsigned long long o =
                (static_cast<unsigned long long>(__reduce_or_sync(0xffffffffu, static_cast<uint32_t>(wo >> 32)))
                 << 32) |
                __reduce_or_sync(0xffffffffu, static_cast<uint32_t>(wo));
            const unsigned long long diff = a ^ o;  // bits in which some keys differ
            const int hb = diff ? 63 - __clzll(static_cast<long long>(diff)) : 0;
            // the first digit is the 11 bits ending at that bit, so every bit it
            // holds can differ (a digit below bit 0 is cut to its bits >= 0)
            const unsigned long long above = hb >= 63 ? 0ull : ~((2ull << hb) - 1);
            if (lane == 0) {
                sh_shift = hb - 10;
                sh_prefix = o & above;  // = a & above
                sh_mask = above;
                sh_k = B;
                sh_ncand = 0;
            }
        }
        for (int i = tid; i < kBins; i += kSelThreads) hist[i] = 0;
        __syncthreads();
        prefix = sh_prefix;
        mask = sh_mask;
        for (int shift = sh_shift; shift > -11; shift -= 11) {
            const int dsh = shift < 0 ? 0 : shift;                                       // the digit's lowest bit
            const unsigned long long dmask = shift < 0 ? (0x7FFull >> -shift) : 0x7FFull;  // its bits, at dsh
            for (int i = tid; i < n; i += kSelThreads) {
                const unsigned long long kk = key[i];
                if ((kk & mask) == prefix) atomicAdd(&hist[(kk >> dsh) & dmask], 1u);
            }
            __syncthreads();
            // the digit of the k-th largest: thread t < 512 owns digits 2047 - 4 t - j
            unsigned c[4] = {0, 0, 0, 0}, local = 0;
            if (tid < kBins / 4) {
                const uint4 h4 = *reinterpret_cast<const uint4*>(hist + kBins - 4 - 4 * tid);
                c[0] = h4.w;
                c[1] = h4.z;
                c[2] = h4.y;
                c[3] = h4.x;
                local = c[0] + c[1] + c[2] + c[3];
            }
            unsigned incl = local;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (lane == 31) warp_sums[tid >> 5] = incl;
            __syncthreads();
            if (tid < kBins / 4) {
                unsigned above = incl - local;
                for (int w = 0; w < (tid >> 5); ++w) above += warp_sums[w];
                const unsigned k = sh_k;
                if (above < k && above + local >= k) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (above < k && above + c[j] >= k) {
                            sh_prefix = prefix | (static_cast<unsigned long long>(kBins - 1 - 4 * tid - j) << dsh);
                            sh_mask = mask | (dmask << dsh);
                            sh_in = c[j];
                            warp_sums[kSelWarps] = k - above;  // read below; sh_k is still being read
                        }
                        above += c[j];
                    }
                }
            }
            __syncthreads();
            prefix = sh_prefix;
            mask = sh_mask;
            const int in = sh_in, k = warp_sums[kSelWarps];
            if (in == k) break;  // every member of the bin is kept (keys are distinct: at the latest
                                 // when no bit is left)
            if (in <= kDirect) {
                // rank the bin's members: the k-th largest is the last one kept
                for (int i = tid; i < n; i += kSelThreads) {
                    const unsigned long long kk = key[i];
                    if ((kk & mask) == prefix) cand[atomicAdd(&sh_ncand, 1)] = kk;
                }
                __syncthreads();
                if (tid < in) {
                    const unsigned long long me = cand[tid];
                    int rank = 0;
                    for (int q = 0; q < in; ++q) rank += cand[q] > me ? 1 : 0;
                    if (rank == k - 1) sh_prefix = me;
                }
                __syncthreads();
                prefix = sh_prefix;
                mask = ~0ull;
                break;
            }
            if (tid == 0) sh_k = k;
            for (int i = tid; i < kBins; i += kSelThreads) hist[i] = 0;
            __syncthreads();
        }
        __syncthreads();
    } else {
        mask = 0;
        prefix = 0;  // every member kept
    }

    // 3. free slots (evicted or empty, ascending) and admitted tokens (ascending):
    // one block scan over both counts, packed as free + (admitted << 16)
    // (at most kMaxPool < 2^16 free slots, and kMaxFrameTokens admitted)
    const int per = (B + kSelThreads - 1) / kSelThreads;
    const int tper = (T + kSelThreads - 1) / kSelThreads;
    int local_free = 0, local_adm = 0;
    for (int s = tid * per; s < min(B, (tid + 1) * per); ++s)
        local_free += (s >= count || (key[s] & mask) < prefix) ? 1 : 0;
    for (int t = tid * tper; t < min(T, (tid + 1) * tper); ++t)
        local_adm += ((key[count + t] & mask) >= prefix) ? 1 : 0;
    int excl;
    const int tot = block_exclusive_scan(local_free + (local_adm << 16), warp_sums, excl);
    const int nfree = tot & 0xFFFF, nadm = tot >> 16;
    int slot_rank = excl & 0xFFFF, tok_rank = excl >> 16;
    for (int s = tid * per; s < min(B, (tid + 1) * per); ++s)
        if (s >= count || (key[s] & mask) < prefix) {
            if (slot_rank < T) free_slot[slot_rank] = s;
            ++slot_rank;
        }
    for (int t = tid * tper; t < min(T, (tid + 1) * tper); ++t)
        if ((key[count + t] & mask) >= prefix) adm_tok[tok_rank++] = t;
    __syncthreads();
    const int npairs = min(nadm, nfree);
    if (tid == 0 && nadm > nfree) *reinterpret_cast<volatile int32_t*>(p.status) = DEV_BAD_SELECT;

    // 4. gather: 16-byte vector copies of the admitted K and V rows, kGatherBatch of a
    // thread's loads in flight before its first store (196 rows of 256 bytes twice
    // are ten copies per thread: one at a time, each waits for its load)
    constexpr int kGatherBatch = 8;
    const int cs = D == 128 ? 4 : 3, chunks = 1 << cs;  // 16-byte chunks per row
    const size_t src_stride = static_cast<size_t>(p.Hkv) * D;
    const __nv_bfloat16* ksrc = p.k + (static_cast<size_t>(u) * T * p.Hkv + hkv) * D;
    const __nv_bfloat16* vsrc = p.v + (static_cast<size_t>(u) * T * p.Hkv + hkv) * D;
    __nv_bfloat16* kdst = p.state_k + head * B * D;
    __nv_bfloat16* vdst = p.state_v + head * B * D;
    for (int w0 = tid; w0 < npairs << (cs + 1); w0 += kGatherBatch * kSelThreads) {
        uint4 x[kGatherBatch];
#pragma unroll
        for (int e = 0; e < kGatherBatch; ++e) {  // copy w: chunk w % chunks of K (even) or V (odd) of a pair
            const int w = w0 + e * kSelThreads, i = w >> (cs + 1);
            if (i < npairs)
                x[e] = *reinterpret_cast<const uint4*>((((w >> cs) & 1) ? vsrc : ksrc) + adm_tok[i] * src_stride +
                                                       (w & (chunks - 1)) * 8);
        }
#pragma unroll
        for (int e = 0; e < kGatherBatch; ++e) {
            const int w = w0 + e * kSelThreads, i = w >> (cs + 1);
            if (i >= npairs) break;
            const int s = free_slot[i];
            if (!SKV_CHECK(adm_tok[i] >= 0 && adm_tok[i] < T && s >= 0 && s < B, p.status, 2)) continue;
            *reinterpret_cast<uint4*>((((w >> cs) & 1) ? vdst : kdst) + static_cast<size_t>(s) * D +
                                      (w & (chunks - 1)) * 8) = x[e];
        }
    }
    for (int i = tid; i < npairs; i += kSelThreads)
        if (SKV_CHECK(free_slot[i] >= 0 && free_slot[i] < B, p.status, 3)) pos[free_slot[i]] = L + adm_tok[i];
    if (tid == 0) p.counts[head] = min(B, count + T);
    finish_unit(p, u, nf);
}

// K4: D[hkv][L + t][:] = K[t][hkv][:] (and V), one 16-byte chunk per thread.
__global__ void __launch_bounds__(256) decode_cache_append(const AppendParams p)
{
    const int chunks = p.D / 8;
    const long long per_unit = static_cast<long long>(p.T) * p.Hkv * chunks;
    const long long total = 2ll * p.U * per_unit;
    for (long long w = blockIdx.x * 256ll + threadIdx.x; w < total; w += 256ll * gridDim.x) {
        const int which = static_cast<int>(w / (p.U * per_unit));
        const long long r = w % (p.U * per_unit);
        const int u = static_cast<int>(r / per_unit);
        const long long rr = r % per_unit;  // source order [t][hkv][chunk]
        const int t = static_cast<int>(rr / (p.Hkv * chunks));
        const int hkv = static_cast<int>((rr / chunks) % p.Hkv);
        const int ch = static_cast<int>(rr % chunks);
        const int ua = p.units.unit_abs(u);
        const size_t head = static_cast<size_t>(ua) * p.Hkv + hkv;
        const long long row = static_cast<long long>(p.frames[head]) * p.row_mul +
                              (p.row_add ? p.row_add[head] : 0) + t;
        const __nv_bfloat16* src = (which ? p.v : p.k) + static_cast<size_t>(u) * per_unit * 8 +
                                   static_cast<size_t>(rr) * 8;
        __nv_bfloat16* dst = (which ? p.cache_v : p.cache_k) +
                             (head * p.cap + row) * p.D + ch * 8;
        if (!SKV_CHECK(row >= 0 && row < p.cap, p.status, 4)) continue;
        *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(src);
    }
}

// one CTA of kGuardBytes threads per guard band
__global__ void canary_check(const uint8_t* arena, const GuardList g, int32_t* status)
{
    const int b = blockIdx.x;
    if (b < g.n && arena[g.off[b] + threadIdx.x] != kGuardFill)
        *reinterpret_cast<volatile int32_t*>(status) = DEV_CANARY | (b << 8);
}

}  // namespace

cudaError_t launch_canary_check(const uint8_t* arena, const GuardList& g, int32_t* status, cudaStream_t st)
{
    if (g.n <= 0) return cudaSuccess;
    canary_check<<<g.n, kGuardBytes, 0, st>>>(arena, g, status);
    return cudaGetLastError();
}

size_t select_smem_bytes(int P, int T)
{
    return (static_cast<size_t>(P) * 8 + 15) / 16 * 16 +
           std::max(static_cast<size_t>(T) * 8, static_cast<size_t>(kDirect * 8 + kBins * 4));
}

cudaError_t select_prepare()
{
    const int bytes = static_cast<int>(select_smem_bytes(kMaxPool, kMaxFrameTokens));
    for (auto kernel : {state_select_gather<true, kMem, int>, state_select_gather<false, kMem, int>,
                        state_select_gather<false, kMemFewTiles, int>, state_select_gather<false, kMem, long long>}) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// CTAs per head: a power of two up to 8 (the portable cluster size) that leaves each
// a full round of its threads (four columns each, or two members), while the heads'
// CTAs take three quarters of the SMs or fewer.  The cluster's barriers and remote
// stores cost ~1.3 us, a round of columns is ~0.5, of members ~1.3, and with
// layer-level scores each is Hkv + 1 sums: hence the five rounds for plain columns.
// Per frame of one 7B layer, on one CTA and split: pool 2797 (members) 34.3 -> 33.2
// us, 5317 (members) 47.6 -> 44.7, 8388 layer-level 70.7 -> 61.9, 16,580 89.9 ->
// 88.6; columns at 5316 and 8388 would be 45.9 -> 46.7 and 57.0 -> 57.3.
int select_split(const SelectParams& p, int U)
{
    const long long heads = static_cast<long long>(U) * p.Hkv, sms = device_sm_count();
    const bool columns = (p.P & 3) == 0;
    const int rounds = p.P / ((columns ? 4 : kMem) * kSelThreads);
    int C = 1;
    if (columns && !p.shared && rounds < 5) return C;
    while (C < kMaxSelSplit && 2 * C <= rounds && heads * 2 * C * 4 <= sms * 3) C *= 2;
    return C;
}

cudaError_t launch_select(const SelectParams& p, int U, cudaStream_t st)
{
    if (U <= 0) return cudaSuccess;
    SelectParams q = p;
    q.U = U;
    q.split = select_split(p, U);
    q.appenders = append_ctas(p.T, p.Hkv, p.D, q.split);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(static_cast<unsigned>(U) * (p.Hkv * q.split + q.appenders));
    cfg.blockDim = dim3(kSelThreads);
    cfg.dynamicSmemBytes = select_smem_bytes(p.P, p.T);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = q.split;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = q.split > 1 ? 2 : 1;
    // (thousands of heads, as the 64-bit append takes, are never split)
    const auto kernel = q.split > 1                             ? state_select_gather<true, kMem, int>
                        : !append_narrow(p.T, p.Hkv, p.D)       ? state_select_gather<false, kMem, long long>
                        : select_members(p) == kMemFewTiles     ? state_select_gather<false, kMemFewTiles, int>
                                                                : state_select_gather<false, kMem, int>;
    return cudaLaunchKernelEx(&cfg, kernel, q);
}

// Recency window (the baseline the method is compared with): the state keeps
// the B most recent tokens.  Token t of frame n sits at position (n-1) T + t
// and goes to ring slot position mod B, which holds the token B positions
// older -- exactly the one leaving the window -- so no search is needed.
// A flat grid of 16-byte row chunks (like the cache append); a second kernel
// then advances the per-head counters, after every copy has read them.
__global__ void __launch_bounds__(256) state_recency_scatter(const RecencyParams p)
{
    const int t0 = p.T > p.B ? p.T - p.B : 0;  // older frame tokens leave the window at once
    const int nt = p.T - t0, chunks = p.D / 8;
    const long long per_head = static_cast<long long>(nt) * (chunks + 1);  // rows x (chunks + position)
    const long long total = 2ll * p.U * p.Hkv * per_head;
    for (long long w = blockIdx.x * 256ll + threadIdx.x; w < total; w += 256ll * gridDim.x) {
        const int which = static_cast<int>(w / (p.U * p.Hkv * per_head));
        const long long r = w % (p.U * p.Hkv * per_head);
        const int uh = static_cast<int>(r / per_head);
        const int u = uh / p.Hkv, hkv = uh % p.Hkv;
        const long long rr = r % per_head;
        const int t = t0 + static_cast<int>(rr / (chunks + 1));
        const int ch = static_cast<int>(rr % (chunks + 1));
        const size_t head = static_cast<size_t>(p.units.unit_abs(u)) * p.Hkv + hkv;
        const long long pos = static_cast<long long>(p.frames[head]) * p.T + t;
        const long long slot = pos % p.B;
        if (ch == chunks) {  // one thread per row writes its position
            if (which == 0) p.positions[head * p.B + slot] = static_cast<int32_t>(pos);
            continue;
        }
        const __nv_bfloat16* src =
            (which ? p.v : p.k) + ((static_cast<size_t>(u) * p.T + t) * p.Hkv + hkv) * p.D + ch * 8;
        __nv_bfloat16* dst = (which ? p.state_v : p.state_k) + (head * p.B + slot) * p.D + ch * 8;
        *reinterpret_cast<uint4*>(dst) = *reinterpret_cast<const uint4*>(src);
    }
}

__global__ void recency_advance(const RecencyParams p)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= p.U * p.Hkv) return;
    const size_t head = static_cast<size_t>(p.units.unit_abs(i / p.Hkv)) * p.Hkv + i % p.Hkv;
    const long long seen = static_cast<long long>(p.frames[head] + 1) * p.T;
    p.counts[head] = static_cast<int32_t>(seen < p.B ? seen : p.B);
    p.frames[head] += 1;
}

cudaError_t launch_recency(const RecencyParams& p, cudaStream_t st)
{
    if (p.B > 0) {
        const int t0 = p.T > p.B ? p.T - p.B : 0;
        const long long work = 2ll * p.U * p.Hkv * (p.T - t0) * (p.D / 8 + 1);
        const int blocks = static_cast<int>(std::min<long long>((work + 255) / 256, 152ll * 16));
        state_recency_scatter<<<blocks, 256, 0, st>>>(p);
    }
    recency_advance<<<(p.U * p.Hkv + 255) / 256, 256, 0, st>>>(p);
    return cudaGetLastError();
}

__global__ void advance_counter(int32_t* counter, UnitRange units, int U, int Hkv, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= U * Hkv) return;
    counter[static_cast<size_t>(units.unit_abs(i / Hkv)) * Hkv + i % Hkv] += n;
}

cudaError_t launch_advance(int32_t* counter, UnitRange units, int U, int Hkv, int n,
                           cudaStream_t st)
{
    advance_counter<<<(U * Hkv + 255) / 256, 256, 0, st>>>(counter, units, U, Hkv, n);
    return cudaGetLastError();
}

cudaError_t launch_append(const AppendParams& p, cudaStream_t st)
{
    const long long total = 2ll * p.U * p.T * p.Hkv * (p.D / 8);
    const long long blocks = (total + 255) / 256;
    const int grid = static_cast<int>(blocks < 152ll * 64 ? blocks : 152ll * 64);
    decode_cache_append<<<grid, 256, 0, st>>>(p);
    return cudaGetLastError();
}

}  // namespace statekv
