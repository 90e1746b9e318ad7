// K1: frame attention with saved log-sum-exp and fused importance partials.
//
// A work unit is 128 query rows of one KV-head group of one (stream, layer).
// Rows are packed token-major, row r = t * G + g (query head hkv*G + g of
// token t), so a tile covers ~128/G consecutive tokens and the in-frame
// causal mask of Eq. 5 skips every frame-key tile beyond its last token.
//
// Keys are the valid state slots (tiles of 128 from the compressed state)
// followed by the frame's tokens.  Two passes over the key tiles (App. B.1):
//   pass A  S = Q K^T  -> online max / sum per row -> log-sum-exp
//   pass B  S = Q K^T  -> P = exp(S - LSE) (fp32) -> column sums of P over the
//           tile's 128 rows (Eq. 1's importance, restricted to these rows) and
//           O += P V with P in bf16.
// tcgen05 runs every contraction with the A operand in TMEM (Q for Q K^T, P
// for P V), so each MMA streams only K or V from shared memory.
//
// K and V tiles of 128 keys stream through a ring of six 32 KB shared-memory
// slots in one sequence, pass A's K tiles, then pass B's K(0) V(0) K(1) V(1) ...;
// a slot is refilled once the MMAs that read it have completed (their commit
// arrives on the slot's barrier).  The work on a tile goes in steps of 64 keys,
// its halves: a step's scores get one of five TMEM buffers of 64 columns, and
// its P overwrites the first half of them.  So up to five steps of each pass are
// under way at once, in different stages: Q K^T, exponentials, P V.
//
// The kernel is persistent: one CTA per SM walks work units (query tile, KV
// head, unit) in a fixed stride.  Ring, TMEM and barriers carry over from one
// unit to the next, so the producer loads the next unit's first tiles while
// the current one finishes, and its first Q K^T run while the previous O is
// read out.
//
// 512 threads, four warpgroups:
//   WG0  warp 0 producer (TMA), warps 1 and 3 MMA issuers X and Y (warp 1
//        also owns TMEM), warp 2 the column-sum reducer.  Pass A: X issues the
//        Q K^T of even steps, Y of odd ones; pass B: X every Q K^T, Y every P V
//        (in order, so O accumulates deterministically).
//   WG1..3  softmax warpgroups; they take the steps in turn.  Pass A: thread =
//        query row, running max and sum.  Pass B: a thread holds 4 rows x 16
//        columns, so the column sums start in registers.
// What bounds it: no single unit.  At the 28-layer 7B stack (1232 units of ~35
// steps, 213 us) the tensor core is busy 56% of the time, and taking out the
// MMAs, the exponentials or the copies each saves 20 to 30 us: a step's chain
// (barrier, TMEM load, 64 exponentials per thread, P store, column sums,
// barrier) is ~1.2k cycles in a warpgroup against 540 of MMA in pass B.  Three
// warpgroups on separate steps keep their phases apart; two on halves of one
// tile (both in the same phase, and the odd tiles' Q K^T waiting for the P V
// that read their P) and four (104 registers) were slower.  What had bound it
// before was the issue of the MMAs and copies by one lane of a divergent warp;
// see umma_ts.  Measured per frame, that form and this one (attention and
// selection): 28-layer 7B stack 267 -> 228 us, 80-layer 72B stack 2.79 -> 2.47
// ms, 28 layers over 32 frames of exact attention 622 -> 548 us.
//
// Few units (one layer of a 7B model has 44 for 152 SMs): the split form.  A
// thread-block cluster of S CTAs shares a unit, each CTA with a run of its key
// tiles: pass A over them, then the CTAs exchange their rows' (max, sum) in
// distributed shared memory, pass B over the same tiles (the importance columns
// are its own), and last the S partial O are added in rank order, each CTA
// finishing 1/S of the rows.  Per frame (attention and selection): one 7B layer (15
// key tiles, S = 3) 35.2 -> 32.5 us, with a state of 16,384 (130 tiles) 184 ->
// 111 us.
// Every mbarrier wait is bounded by the watchdog; on expiry the CTA records
// DEV_TIMEOUT_ATTN, drains its in-flight copies and MMAs, frees TMEM and exits.
#include "sm103_ptx.cuh"
#include "statekv_kernels.cuh"

namespace statekv {
namespace {

using namespace ptx;

constexpr int kWG = 3;                    // softmax warpgroups
constexpr int kSoftThreads = 128 * kWG;
constexpr int kThreads = 128 + kSoftThreads;
constexpr int kSlots = 6;        // 32 KB K/V tile slots (D = 128), one ring
constexpr int kStep = 64;        // keys per step: half a K/V tile
constexpr int kMaxSplit = 8;     // CTAs that may share a unit (the portable cluster size)
constexpr int kBufs = 5;         // score buffers
// TMEM columns: Q [0, 64) | O [64, 192) | five score buffers of 64 columns.
// A step's P (bf16 pairs) overwrites the first 32 columns of its own scores.
constexpr uint32_t kColO = 64;
constexpr uint32_t kColS = 192;
// Barriers of a step are indexed by step mod 10, so that each waiter has seen the
// barrier's previous phase and can never mistake a phase two back for the one it
// waits for (two issuers and kWG warpgroups take steps in turn).
constexpr int kBars = 2 * kBufs;
constexpr int kWgArrive = 128;   // arrivals of a warpgroup on a barrier: every thread (one per warp was slower)

template <int D>
struct AttnLayout {
    static constexpr int kTileBytes = kBN * D * 2;  // one K or V tile
    static constexpr int kOffSlots = 0;
    // column sums of four pass-B steps: float[4][4 warps][32 lanes][2]
    static constexpr int kOffStage = kOffSlots + kSlots * kTileBytes;
    static constexpr int kOffStat = kOffStage + 4 * 4 * 32 * 2 * 4;  // float[kWG][2][128]
    static constexpr int kOffXStat = kOffStat + kWG * 2 * kBM * 4;  // split form: float2[8 ranks][128]
    static constexpr int kOffBar = kOffXStat + kMaxSplit * kBM * 8;
    static constexpr int kOStageLd = D + 4;  // split form: O staged over the ring, rows padded by a float4
    static_assert(kBM * kOStageLd * 4 <= kSlots * kTileBytes, "O staging");
    // slot_full[6] slot_empty[6] s_full[10] s_free[10] p_full[8] stage_full[4]
    // stage_free[4] q_full o_full o_read drain stall
    static constexpr int kNumBars = 2 * kSlots + 2 * kBars + 8 + 8 + 5;
    static constexpr int kOffMisc = kOffBar + kNumBars * 8;
    static constexpr int kBytes = kOffMisc + 16;
    static constexpr int kAlloc = kBytes + 1024;  // room to align the base to 1 KB
    static_assert(kOffSlots % 1024 == 0 && kTileBytes % 1024 == 0, "align");
    static_assert(kAlloc <= 232448, "shared memory budget");
};

__device__ __forceinline__ float ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float max3(float a, float b, float c)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Packed pair of floats in one 64-bit register (sm_100+ f32x2 arithmetic).
struct f2 {
    uint64_t r;
};

__device__ __forceinline__ f2 pk(float lo, float hi)
{
    f2 o;
    asm("mov.b64 %0, {%1, %2};" : "=l"(o.r) : "f"(lo), "f"(hi));
    return o;
}

__device__ __forceinline__ void upk(f2 x, float& lo, float& hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(x.r));
}

__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c)
{
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d.r) : "l"(a.r), "l"(b.r), "l"(c.r));
    return d;
}

__device__ __forceinline__ f2 add2(f2 a, f2 b)
{
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d.r) : "l"(a.r), "l"(b.r));
    return d;
}

__device__ __forceinline__ void named_bar_sync(int id, int nthreads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

__device__ __forceinline__ void named_bar_arrive(int id, int nthreads)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// A position in a cycle of N places (ring slots, score buffers) and the parity of
// its current use.
template <uint32_t N>
struct Cycle {
    uint32_t at, ph;
    __device__ __forceinline__ Cycle plus(uint32_t n) const  // any n
    {
        const uint32_t t = at + n, q = t / N;
        return Cycle{t - q * N, ph ^ (q & 1)};
    }
    __device__ __forceinline__ void step(uint32_t n)  // n <= N
    {
        at += n;
        if (at >= N) {
            at -= N;
            ph ^= 1;
        }
    }
};

// 16 consecutive 32-bit TMEM columns of this thread's lane <- registers.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0],"
        " {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]),
        "r"(r[15])
        : "memory");
}

__device__ __forceinline__ void tmem_st_wait()
{
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// 16 TMEM lanes x 64 columns -> 32 registers (.16x256b layout): register
// 4r + 2k + e holds lane (base + t/4 + 8k), column 8r + 2(t%4) + e, r < 8.
__device__ __forceinline__ void tmem_ld_16x256b_x8(uint32_t taddr, float (&v)[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x8.b32"
        " {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15,"
        " %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31},"
        " [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// 16 registers -> 16 TMEM lanes x 32 columns (.16x128b layout): register
// 2r + k goes to lane (base + t/4 + 8k), column 4r + t%4, r < 8.
__device__ __forceinline__ void tmem_st_16x128b_x8(uint32_t taddr, const uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.16x128b.x8.b32 [%0],"
        " {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]),
        "r"(r[15])
        : "memory");
}

// Sums over the 8 lanes that share lane % 4 (lane bits 2..4) of 16 values,
// as a reduce-scatter: lane l returns the sums of values 2 (l/4) and 2 (l/4) + 1.
__device__ __forceinline__ float2 lane8_reduce_scatter(float (&x)[16], int lane)
{
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const bool up = (lane & 16) != 0;
        const float send = up ? x[i] : x[i + 8];
        const float keep = up ? x[i + 8] : x[i];
        x[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool up = (lane & 8) != 0;
        const float send = up ? x[i] : x[i + 4];
        const float keep = up ? x[i + 4] : x[i];
        x[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
    float2 out;
    {
        const bool up = (lane & 4) != 0;
        const float s0 = up ? x[0] : x[2], k0 = up ? x[2] : x[0];
        const float s1 = up ? x[1] : x[3], k1 = up ? x[3] : x[1];
        out.x = k0 + __shfl_xor_sync(0xffffffffu, s0, 4);
        out.y = k1 + __shfl_xor_sync(0xffffffffu, s1, 4);
    }
    return out;
}

// One work unit: the 128 query rows of tile mt of KV head hkv of the call's
// unit u, with the key range the unit sees.  Units are numbered with the tile
// fastest, then the KV head, then the unit.  Keys are taken in steps of 64: the
// state's (or cache's) first, then the frame's, each range starting a new tile.
struct WorkUnit {
    int mt, hkv, u, ua;
    int count;  // visible keys before the frame (state slots or cache rows)
    int nfull;  // whole 128-key tiles over them
    int nss;    // steps over them
    int nst;    // tiles over them
    int nfs;    // frame steps the tile's last row can see
    int s0, t0; // this CTA's first step and tile (0 unless it shares the unit)
    int ns;     // and how many of each it takes
    int nt;
    int rot;    // first state tile (see state_tile)
};

template <bool kSplit>
__device__ __forceinline__ WorkUnit work_unit(const AttnParams& p, int w)
{
    WorkUnit x;
    x.mt = w % p.MT;
    const int r = w / p.MT;
    x.hkv = r % p.Hkv;
    x.u = r / p.Hkv;
    x.ua = p.units.unit_abs(x.u);
    const int head = x.ua * p.Hkv + x.hkv;
    x.count = p.count_mul * ((p.B > 0 || p.count_mul > 1) ? p.counts[head] : 0) +
              (p.count_add ? p.count_add[head] : 0);
    x.nfull = x.count / kBN;
    x.nss = (x.count + kStep - 1) / kStep;
    x.nst = (x.count + kBN - 1) / kBN;
    const int row_hi = min(p.G * p.T, (x.mt + 1) * kBM) - 1;
    x.nfs = p.causal ? (row_hi / p.G) / kStep + 1 : (p.T + kStep - 1) / kStep;
    x.s0 = x.t0 = 0;
    x.ns = x.nss + x.nfs;
    x.nt = x.nst + (x.nfs + 1) / 2;
    if (kSplit) {  // rank r of S takes tiles [nt r / S, nt (r + 1) / S)
        const int r = static_cast<int>(cluster_ctarank()), nt = x.nt, ns = x.ns;
        auto first_step = [&](int t) { return t >= nt ? ns : t <= x.nst ? min(2 * t, x.nss) : x.nss + 2 * (t - x.nst); };
        const int t1 = nt * (r + 1) / p.split;
        x.t0 = nt * r / p.split;
        x.s0 = first_step(x.t0);
        x.nt = t1 - x.t0;
        x.ns = first_step(t1) - x.s0;
    }
    // The query tiles of one KV head read the same state tiles; each starts at
    // a different whole one (a fixed rotation) so they do not all request the
    // same L2 lines at the same moment.  The ragged tile comes last; frame
    // tiles keep their order.
    x.rot = x.nfull > 0 ? (x.mt * 3) % x.nfull : 0;
    return x;
}

// the state tile taken t-th
__device__ __forceinline__ int state_tile(const WorkUnit& x, int t)
{
    return t >= x.nfull ? t : t + x.rot < x.nfull ? t + x.rot : t + x.rot - x.nfull;
}

// The first key of step s: state slot / cache row (s < nss) or frame token.
__device__ __forceinline__ int step_key(const WorkUnit& x, int s)
{
    return s < x.nss ? state_tile(x, s >> 1) * kBN + (s & 1) * kStep : (s - x.nss) * kStep;
}

constexpr int kAuxRegs = 80;    // registers per thread of the first warpgroup
constexpr int kSoftRegs = 144;  // and of the softmax warpgroups

// The same for a whole warp, every field the same register for all lanes as far as
// the compiler can tell (it comes through a shuffle).
template <bool kSplit>
__device__ __forceinline__ WorkUnit work_unit_uniform(const AttnParams& p, int w)
{
    WorkUnit x = work_unit<kSplit>(p, w);
    x.hkv = uniform(x.hkv);
    x.u = uniform(x.u);
    x.ua = uniform(x.ua);
    x.nfull = uniform(x.nfull);
    x.rot = uniform(x.rot);
    x.nss = uniform(x.nss);
    x.nst = uniform(x.nst);
    x.nfs = uniform(x.nfs);
    x.s0 = kSplit ? uniform(x.s0) : 0;
    x.t0 = kSplit ? uniform(x.t0) : 0;
    x.ns = uniform(x.ns);
    x.nt = uniform(x.nt);
    return x;
}

// Persistent: one CTA per SM walks the work units w = blockIdx.x, + gridDim.x,
// ...  The ring, the TMEM allocation and every barrier live across units: the
// producer loads the next unit's first tiles while the current one finishes.
// Steps are numbered through the CTA's life: a unit with first step gb takes
// gb .. gb + ns - 1 in pass A and gb + ns .. gb + 2 ns - 1 in pass B, step g uses
// score buffer g % 5 and belongs to warpgroup g % kWG; the ring holds the unit's nt
// K tiles, then K V K V ...; pb counts pass-B steps.
// The split form's CTA has one unit, blockIdx.x / S.
template <int D, bool kSplit>
__global__ void __launch_bounds__(kThreads, 1)
    frame_attn_lse_importance(const __grid_constant__ CUtensorMap tm_sk,
                              const __grid_constant__ CUtensorMap tm_sv,
                              const __grid_constant__ CUtensorMap tm_fk,
                              const __grid_constant__ CUtensorMap tm_fv, const AttnParams p)
{
    using L = AttnLayout<D>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
    uint8_t* sSlot = sm + L::kOffSlots;
    float2* stage = reinterpret_cast<float2*>(sm + L::kOffStage);
    float* stat = reinterpret_cast<float*>(sm + L::kOffStat);
    float2* xstat = reinterpret_cast<float2*>(sm + L::kOffXStat);
    uint64_t* bars = reinterpret_cast<uint64_t*>(sm + L::kOffBar);
    uint64_t* slot_full = bars;                 // ring slot loaded
    uint64_t* slot_empty = slot_full + kSlots;  // the MMAs of its steps have read it (2 arrivals)
    uint64_t* s_full = slot_empty + kSlots;     // Q K^T of step g done (index g % 10)
    uint64_t* s_free = s_full + kBars;          // step g's buffer free: pass A read, pass B P V done
    uint64_t* p_full = s_free + kBars;          // P of pass-B step pb written (index pb % 8)
    uint64_t* stage_full = p_full + 8;          // column sums of pass-B step pb staged (index pb % 4)
    uint64_t* stage_free = stage_full + 4;      // and read by the reducer warp
    uint64_t* q_full = stage_free + 4;          // per unit: Q is in TMEM
    uint64_t* o_full = q_full + 1;              // per unit: every P V has completed
    uint64_t* o_read = q_full + 2;              // per unit: O has been read out of TMEM
    uint64_t* drain = q_full + 3;
    uint64_t* stall = q_full + 4;               // watchdog self-test: never completed
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + L::kOffMisc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + L::kOffMisc + 4);

    // barrier i of the order above at bar0 + 8 i
    const uint32_t bar0 = smem_addr(bars);
    constexpr uint32_t kBarSlotFull = 0, kBarSlotEmpty = 8 * kSlots, kBarSFull = 16 * kSlots,
                       kBarSFree = kBarSFull + 8 * kBars, kBarPFull = kBarSFree + 8 * kBars,
                       kBarStageFull = kBarPFull + 64, kBarStageFree = kBarStageFull + 32,
                       kBarQFull = kBarStageFree + 32, kBarOFull = kBarQFull + 8, kBarORead = kBarQFull + 16,
                       kBarDrain = kBarQFull + 24, kBarStall = kBarQFull + 32;
    const int warp = uniform(threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const int T = p.T, G = p.G, B = p.B;
    const int rows = G * T;
    const int W = p.MT * p.Hkv * p.U;
    const int w0 = kSplit ? blockIdx.x / p.split : blockIdx.x, wstep = kSplit ? W : gridDim.x;

    // A softmax thread's part of its Q row of unit w (thread 128 + i: warpgroup
    // i / 128, row i % 128; warpgroup wg < 2 holds d in [64 wg, 64 (wg + 1))).
    // Padding rows load the last row (zeroed when they are stored).
    uint4 qreg[8];
    auto q_src = [&](int w) -> const uint4* {
        const int tq = static_cast<int>(threadIdx.x) - 128, qwg = tq >> 7;
        if (p.q == nullptr || w >= W || tq < 0 || qwg * 64 >= D) return nullptr;  // nothing to load
        const int mt = w % p.MT, r = w / p.MT, hkv = r % p.Hkv, u = r / p.Hkv;
        const int qr = min(mt * kBM + (tq & 127), rows - 1), t = qr / G, g = qr - t * G;
        return reinterpret_cast<const uint4*>(
            p.q + ((static_cast<size_t>(u) * T + t) * p.Hq + hkv * G + g) * D + qwg * 64);
    };
    auto load_q = [&](int w) {
        const uint4* src = q_src(w);
#pragma unroll
        for (int i = 0; i < 8; ++i) qreg[i] = make_uint4(0u, 0u, 0u, 0u);
        if (src)
#pragma unroll
            for (int i = 0; i < 8; ++i) qreg[i] = src[i];
    };
    auto prefetch_q = [&](int w) {
        const uint4* src = q_src(w);
        if (src) asm volatile("prefetch.global.L2 [%0];" ::"l"(src));
    };
    if (threadIdx.x == 0) {
        for (int i = 0; i < kSlots; ++i) {
            mbar_init(&slot_full[i], 1);
            mbar_init(&slot_empty[i], 2);
        }
        for (int i = 0; i < kBars; ++i) {
            mbar_init(&s_full[i], 1);
            mbar_init(&s_free[i], kWgArrive);
        }
        for (int i = 0; i < 8; ++i) mbar_init(&p_full[i], kWgArrive);
        for (int i = 0; i < 4; ++i) {
            mbar_init(&stage_full[i], kWgArrive);
            mbar_init(&stage_free[i], 1);
        }
        mbar_init(q_full, kSoftThreads);
        mbar_init(o_full, 1);
        mbar_init(o_read, kSoftThreads);
        mbar_init(drain, 2);   // one commit per MMA issuer
        mbar_init(stall, 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    // Launched programmatically: everything above overlaps the end of the stream's
    // previous kernel, and nothing it wrote is read before this wait.  Then the next
    // kernel (the selection) may come in as SMs fall idle.
    pdl_wait();
    pdl_launch_dependents();
    load_q(w0);  // the first unit's rows
    __syncthreads();
    // Split form: every thread of the cluster passes four phases of its barrier, on
    // every path: 0 all CTAs run, 1 row statistics exchanged, 2 O staged, 3 O read.
    if (kSplit) cluster_sync();
    tc_fence_after();
    const uint32_t tbase = *tmem_slot;

    // Records an expired wait: DEV_TIMEOUT_ATTN with the waiting site in bits
    // 8..15 (see DeviceError), and tells every role to stop.
    auto fail = [&](int site) {
        if (atomicExch(const_cast<int*>(abort_flag), 1) == 0)  // first failure in the CTA
            *reinterpret_cast<volatile int32_t*>(p.status) = DEV_TIMEOUT_ATTN | (site << 8);
    };

    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kAuxRegs) : "memory");
        if (kSplit) cluster_arrive();  // phase 1: nothing of this warpgroup's to wait for
        if (warp == 0) {
            // ------------------------------------------------------------ producer
            // One ring of tiles for both passes of every unit: per unit, pass A's
            // K tiles, then pass B's K(0) V(0) K(1) V(1) ...  Like the issuers, the whole
            // warp runs the loop and elects a lane for the copies.
            if (elect_one()) {
                tma_prefetch_desc(&tm_fk);
                tma_prefetch_desc(&tm_fv);
                if (B > 0) {
                    tma_prefetch_desc(&tm_sk);
                    tma_prefetch_desc(&tm_sv);
                }
            }
            __syncwarp();
            bool ok = true;
            // the self-test's wait gives up at half the watchdog, so it is
            // deterministically the first wait of the launch to expire
            if (p.selftest_stall && !wait_warp(bar0 + kBarStall, 0, globaltimer() + p.watchdog_ns / 2)) {
                if (lane == 0) fail(1);
                ok = false;
            }
            const uint32_t aSlot = uniform(smem_addr(sSlot));
            uint32_t n = 0;            // items so far
            Cycle<kSlots> ring{0, 0};  // the next item's slot
            for (int w = w0; ok && w < W; w += wstep) {
                const WorkUnit x = work_unit_uniform<kSplit>(p, w);
                const unsigned long long deadline = globaltimer() + p.watchdog_ns;
                auto load = [&](const CUtensorMap* map, int c1, int c2, int c3) {
                    if (n >= kSlots && !wait_warp(bar0 + kBarSlotEmpty + 8 * ring.at, ring.ph ^ 1u, deadline)) return false;
                    const uint32_t full = bar0 + kBarSlotFull + 8 * ring.at, dst = aSlot + ring.at * L::kTileBytes;
                    if (elect_one()) {
                        expect_at(full, L::kTileBytes);
#pragma unroll
                        for (int h = 0; h < D / 64; ++h)
                            tma_load_at(dst + h * (kBN * 128), map, full, h * 64, c1, c2, c3);
                    }
                    ++n;
                    ring.step(1);
                    return true;
                };
                // tile t of the unit's keys: rows of the state (or cache), then of the frame
                auto load_tile = [&](int tl, bool v) {
                    const int t = tl + x.t0;
                    return t < x.nst ? load(v ? &tm_sv : &tm_sk, state_tile(x, t) * kBN, x.hkv, x.ua)
                                     : load(v ? &tm_fv : &tm_fk, x.hkv, (t - x.nst) * kBN, x.u);
                };
#pragma unroll 1
                for (int t = 0; ok && t < x.nt; ++t) ok = load_tile(t, false);
#pragma unroll 1
                for (int t = 0; ok && t < x.nt; ++t) ok = load_tile(t, false) && load_tile(t, true);
                if (!ok && lane == 0) fail(2);
                if (__any_sync(0xffffffffu, *abort_flag != 0)) ok = false;
            }
            // let every copy land, and every slot's last tile be read by its MMAs,
            // before the CTA's memory goes away
            const unsigned long long dl = globaltimer() + p.watchdog_ns;
            for (uint32_t i = 0; i < kSlots && i < n; ++i) {  // the last min(n, 6) items
                const Cycle<kSlots> c = ring.plus(2 * kSlots - 1 - i);  // item n - 1 - i (two turns on, same parity)
                wait_warp(bar0 + (ok ? kBarSlotEmpty : kBarSlotFull) + 8 * c.at, c.ph, dl);
            }
        } else if (warp == 2) {
            // ------------------------------------------------------------ column-sum reducer
            // Pass B, per step: each of a warpgroup's four warps stages the column sums
            // of its 32 rows, two columns per lane; they are added in warp order.
            bool ok = true;
            int pb = 0;
            for (int w = w0; ok && w < W && p.partials != nullptr; w += wstep) {
                const WorkUnit x = work_unit<kSplit>(p, w);
                const unsigned long long deadline = globaltimer() + p.watchdog_ns;
                float* part = p.partials + ((static_cast<size_t>(x.u) * p.Hkv + x.hkv) * p.MT + x.mt) * p.P;
                for (int s = 0; s < x.ns; ++s, ++pb) {
                    const float2* area = stage + (pb & 3) * 128 + lane;
                    ok = wait_warp(bar0 + kBarStageFull + 8 * (pb & 3), (pb >> 2) & 1, deadline);
                    if (!ok) {
                        if (lane == 0) fail(13);
                        break;
                    }
                    float2 sum = area[0];
#pragma unroll
                    for (int q = 1; q < 4; ++q) {
                        const float2 y = area[32 * q];
                        sum.x += y.x;
                        sum.y += y.y;
                    }
                    __syncwarp();
                    if (lane == 0) arrive_at(bar0 + kBarStageFree + 8 * (pb & 3));
                    const int sg = s + x.s0;  // the unit's step
                    const bool is_state = sg < x.nss;
                    const int key = step_key(x, sg) + 8 * (lane >> 2) + 2 * (lane & 3);
                    const int lim = is_state ? x.count : T;
                    float* dst = part + (is_state ? 0 : B) + key;
                    if (key < lim) dst[0] = sum.x;
                    if (key + 1 < lim) dst[1] = sum.y;
                }
            }
        } else {
            // ------------------------------------------------------------ MMA issuers
            // Pass A: X (warp 1) takes the even steps' Q K^T, Y (warp 3) the odd ones'.
            // Pass B: X issues every Q K^T, Y every P V, in step order.
            // The whole warp runs the loops, with uniform operands, and elects a lane
            // for each instruction (see umma_ts).
            const bool isx = warp == 1;
            const uint32_t aSlot = uniform(smem_addr(sSlot));
            const uint64_t dk = sdesc_sw128(aSlot, 16, 1024);         // K-major, slot 0
            const uint64_t dv = sdesc_sw128(aSlot, kBN * 128, 1024);  // MN-major, slot 0
            // descriptor address units: a slot, half a tile's rows (64 of K, or 64 keys of V)
            constexpr uint32_t kSlotStep = L::kTileBytes >> 4;
            constexpr uint32_t kHalf = (kStep * 128) >> 4;
            const uint32_t tb0 = uniform(tbase);
            const uint32_t tQ = tb0, tO = tb0 + kColO, tS = tb0 + kColS;
            constexpr uint32_t kIdQK = idesc_bf16_f32(kBM, kStep, false, false);
            constexpr uint32_t kIdPV = idesc_bf16_f32(kBM, D, false, true);
            int site = 4;  // first wait that expired, for the status word
            bool ok = true;
            uint32_t gb = 0, pb = 0, k = 0;  // earlier units' steps, pass-B steps so far, units
            Cycle<kSlots> ring{0, 0};        // the unit's first ring item
            Cycle<kBars> bar{0, 0};          // the unit's first step's barriers; buffer = at % 5
            // S = Q K^T of step g (barriers b; half h of the tile in ring slot) once the
            // step g - 5 has left its buffer
            auto qk = [&](uint32_t g, const Cycle<kBars>& b, uint32_t slot, uint32_t h, unsigned long long deadline) {
                const bool hi = b.at >= kBufs;
                if (g >= kBufs && !wait_warp(bar0 + kBarSFree + 8 * (hi ? b.at - kBufs : b.at + kBufs),
                                             hi ? b.ph : b.ph ^ 1u, deadline))
                    return false;
                tc_fence_after();
                const uint64_t bd = dk + slot * kSlotStep + h * kHalf;
                const uint32_t d = tS + (hi ? b.at - kBufs : b.at) * kStep;
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk)  // 16 KB per 64-wide K half of a tile, 32 B per step
                    umma_ts(d, tQ + 8 * kk, bd + (((kk >> 2) * (kBN * 128) + (kk & 3) * 32) >> 4), kIdQK, kk > 0);
                commit_elect(bar0 + kBarSFull + 8 * b.at);
                return true;
            };
            for (int w = w0; ok && w < W; w += wstep, ++k) {
                const WorkUnit x = work_unit_uniform<kSplit>(p, w);
                const uint32_t nt = x.nt, ns = x.ns;
                // tiles of one step: the ragged state tile and the last frame tile, if odd
                // (counted from this CTA's first; one that is not its own compares unequal)
                const uint32_t odd0 = (x.nss & 1) ? x.nst - 1 - x.t0 : ~0u,
                               odd1 = (x.nfs & 1) ? x.nst + x.nfs / 2 - x.t0 : ~0u;
                const unsigned long long deadline = globaltimer() + p.watchdog_ns;
                site = 4;
                ok = wait_warp(bar0 + kBarQFull, k & 1, deadline);
                {   // pass A: step s of the unit is step gb + s; a tile's steps go to both issuers
                    Cycle<kSlots> r = ring;
                    Cycle<kBars> b = bar;
                    uint32_t g = gb;
#pragma unroll 1
                    for (uint32_t t = 0; ok && t < nt; ++t) {
                        const uint32_t nh = t == odd0 || t == odd1 ? 1 : 2;
                        const uint32_t h = (g & 1) == (isx ? 0u : 1u) ? 0u : 1u;  // this issuer's half
                        if (h < nh) {
                            site = 5;
                            if (!(ok = wait_warp(bar0 + kBarSlotFull + 8 * r.at, r.ph, deadline))) break;
                            site = 6;
                            Cycle<kBars> c = b;
                            c.step(h);
                            if (!(ok = qk(g + h, c, r.at, h, deadline))) break;
                            if (nh == 1 && elect_one()) arrive_at(bar0 + kBarSlotEmpty + 8 * r.at);
                            commit_elect(bar0 + kBarSlotEmpty + 8 * r.at);
                        }
                        g += nh;
                        b.step(nh);
                        r.step(1);
                    }
                }
                Cycle<kBars> b = bar.plus(ns);
                if (isx) {
                    // pass B Q K^T, in step order
                    Cycle<kSlots> r = ring.plus(nt);
                    uint32_t g = gb + ns;
#pragma unroll 1
                    for (uint32_t t = 0; ok && t < nt; ++t) {
                        const uint32_t nh = t == odd0 || t == odd1 ? 1 : 2;
                        site = 5;
                        if (!(ok = wait_warp(bar0 + kBarSlotFull + 8 * r.at, r.ph, deadline))) break;
                        site = 9;
#pragma unroll
                        for (uint32_t h = 0; h < 2; ++h) {
                            if (h >= nh || !ok) break;
                            ok = qk(g, b, r.at, h, deadline);
                            ++g;
                            b.step(1);
                        }
                        if (elect_one()) arrive_at(bar0 + kBarSlotEmpty + 8 * r.at);
                        commit_elect(bar0 + kBarSlotEmpty + 8 * r.at);
                        r.step(2);
                    }
                } else {
                    // O += P V, in step order (O accumulates deterministically)
                    Cycle<kSlots> r = ring.plus(nt + 1);
                    site = 7;
                    if (ok && k >= 1) ok = wait_warp(bar0 + kBarORead, (k - 1) & 1, deadline);
#pragma unroll 1
                    for (uint32_t t = 0; ok && t < nt; ++t) {
                        const uint32_t nh = t == odd0 || t == odd1 ? 1 : 2;
#pragma unroll
                        for (uint32_t h = 0; h < 2; ++h) {
                            if (h >= nh || !ok) break;
                            // P first: once the unit's first P is written every pass-A tile has
                            // landed, so the V slot's barrier is at most one phase behind
                            site = 7;
                            if (!(ok = wait_warp(bar0 + kBarPFull + 8 * (pb & 7), (pb >> 3) & 1, deadline))) break;
                            ++pb;
                            site = 8;
                            if (h == 0 && !(ok = wait_warp(bar0 + kBarSlotFull + 8 * r.at, r.ph, deadline))) break;
                            tc_fence_after();
                            const uint64_t bd = dv + r.at * kSlotStep + h * kHalf;
                            const uint32_t pa = tS + (b.at >= kBufs ? b.at - kBufs : b.at) * kStep;
#pragma unroll
                            for (int kk = 0; kk < kStep / 16; ++kk)  // 2 KB of V per 16 keys
                                umma_ts(tO, pa + 8 * kk, bd + ((kk * 2048) >> 4), kIdPV, t > 0 || h > 0 || kk > 0);
                            if (elect_one()) arrive_at(bar0 + kBarSFree + 8 * b.at, kWgArrive - 1);
                            commit_elect(bar0 + kBarSFree + 8 * b.at);
                            b.step(1);
                        }
                        if (elect_one()) arrive_at(bar0 + kBarSlotEmpty + 8 * r.at);
                        commit_elect(bar0 + kBarSlotEmpty + 8 * r.at);
                        r.step(2);
                    }
                    if (ok) commit_elect(bar0 + kBarOFull);
                }
                gb += 2 * ns;
                ring = ring.plus(3 * nt);
                bar = bar.plus(2 * ns);
            }
            if (!ok && lane == 0) fail(site + (isx ? 0 : 16));
            // Every MMA issued so far must finish before TMEM is released.
            commit_elect(bar0 + kBarDrain);
            wait_warp(bar0 + kBarDrain, 0, globaltimer() + p.watchdog_ns);
        }
        if (kSplit) {
            __syncwarp();
            cluster_wait();  // phase 1
            cluster_sync();  // phase 2
            cluster_sync();  // phase 3
        }
        tc_fence_before();
        __syncthreads();
        if (warp == 1) tmem_dealloc(tbase, 512);
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kSoftRegs) : "memory");
        // ------------------------------------------------------------ softmax warpgroups
        const int wg = (warp >> 2) - 1;
        const int quad = warp & 3;               // TMEM lane quadrant of this warp
        const int row = quad * 32 + lane;        // TMEM lane = query row of the tile
        const uint32_t lane_off = static_cast<uint32_t>(quad * 32) << 16;
        const float c = p.scale_log2;
        const int cq = 2 * (lane & 3);           // this thread's column offset in 8
        const uint32_t tSw = tbase + lane_off + kColS;   // this warp's lanes of the score buffers
        float2* mystage = stage + quad * 32 + lane;  // area i at + 128 i
        const f2 cc = pk(c, c);

        // O rows of unit x -> bf16 out; warpgroup wg < 2 stores columns [wg D/2, (wg + 1) D/2)
        constexpr int kOc = D / 2;
        auto store_o = [&](const WorkUnit& x) {
            if (wg * kOc >= D) return;
            const int my_r = x.mt * kBM + row;
            __nv_bfloat16* dst = p.out;
            if (my_r < rows) {
                const int t = my_r / G, g = my_r - t * G;
                dst += ((static_cast<size_t>(x.u) * T + t) * p.Hq + x.hkv * G + g) * D;
            }
#pragma unroll
            for (int cc2 = 0; cc2 < kOc / 32; ++cc2) {
                const int col = wg * kOc + cc2 * 32;
                float o[32];
                tmem_ld32(tbase + lane_off + kColO + col, o);
                tmem_ld_wait();
                if (my_r < rows) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const uint4 v4 = make_uint4(
                            pack_bf16x2(o[e * 8 + 0], o[e * 8 + 1]), pack_bf16x2(o[e * 8 + 2], o[e * 8 + 3]),
                            pack_bf16x2(o[e * 8 + 4], o[e * 8 + 5]), pack_bf16x2(o[e * 8 + 6], o[e * 8 + 7]));
                        *reinterpret_cast<uint4*>(dst + col + e * 8) = v4;
                    }
                }
            }
        };

        bool ok = true;
        int site = 10;  // first wait that expired, for the status word
        bool exchanged = false;  // split form: past phase 1
        int gb = 0, pbb = 0, k = 0;  // earlier units' steps of both passes, pass-B steps, units
        Cycle<kBars> bar{0, 0};      // the unit's first step's barriers; buffer = at % 5
        WorkUnit prev{};
        for (int w = w0; ok && w < W; w += wstep, ++k) {
            const WorkUnit x = work_unit<kSplit>(p, w);
            const unsigned long long deadline = globaltimer() + p.watchdog_ns;
            const int my_r = x.mt * kBM + row;
            const bool row_valid = my_r < rows;
            const int my_tq = row_valid ? my_r / G : T;  // padding rows see every frame key

            {   // Q row -> TMEM columns [0, D/2) (bf16 pairs).  Every Q K^T of the
                // previous unit has completed (its P V have).
                if (wg * 64 < D) {
                    uint32_t w32[32];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        w32[4 * i] = row_valid ? qreg[i].x : 0u;
                        w32[4 * i + 1] = row_valid ? qreg[i].y : 0u;
                        w32[4 * i + 2] = row_valid ? qreg[i].z : 0u;
                        w32[4 * i + 3] = row_valid ? qreg[i].w : 0u;
                    }
#pragma unroll
                    for (int i = 0; i < 2; ++i)
                        tmem_st16(tbase + lane_off + wg * 32 + 16 * i,
                                  *reinterpret_cast<uint32_t(*)[16]>(&w32[16 * i]));
                    tmem_st_wait();
                }
                tc_fence_before();
                arrive_at(bar0 + kBarQFull);
            }
            if (k >= 1) {  // the previous unit's O, while this unit's first Q K^T run
                store_o(prev);
                tc_fence_before();
                arrive_at(bar0 + kBarORead);
            }

            // ---------------- pass A: online max / sum of exp2 over this warpgroup's steps
            float m = -INFINITY, l = 0.f;  // log2 units, scaled
            const int sA = (wg + kWG - gb % kWG) % kWG;
            Cycle<kBars> b = bar.plus(sA);
            for (int s = sA; s < x.ns; s += kWG) {
                ok = wait_warp(bar0 + kBarSFull + 8 * b.at, b.ph, deadline);
                if (!ok) break;
                tc_fence_after();
                const uint32_t tSa = tSw + (b.at >= kBufs ? b.at - kBufs : b.at) * kStep;
                // the step into registers, then release the buffer at once so
                // the next Q K^T into it can start while this one is reduced
                float v[2][32];
                tmem_ld32(tSa, v[0]);
                tmem_ld32(tSa + 32, v[1]);
                tmem_ld_wait();
                tc_fence_before();
                arrive_at(bar0 + kBarSFree + 8 * b.at);
                b.step(kWG);
                const int sg = s + x.s0;
                if (sg >= 2 * x.nfull) {  // keys [0, lim) of a ragged or frame step are visible to this row
                    const int lim = sg < x.nss ? x.count - sg * kStep
                                               : (p.causal ? min(T, my_tq + 1) : T) - (sg - x.nss) * kStep;
                    if (lim < kStep) {
#pragma unroll
                        for (int ch = 0; ch < 2; ++ch)
#pragma unroll
                            for (int e = 0; e < 32; ++e)
                                v[ch][e] = (ch * 32 + e < lim) ? v[ch][e] : -INFINITY;
                    }
                }
                float mx[4];
#pragma unroll
                for (int q4 = 0; q4 < 4; ++q4) mx[q4] = fmaxf(v[q4 >> 1][(q4 & 1) * 16], v[q4 >> 1][(q4 & 1) * 16 + 1]);
#pragma unroll
                for (int q4 = 0; q4 < 4; ++q4)
#pragma unroll
                    for (int e = 2; e < 16; e += 2)
                        mx[q4] = max3(mx[q4], v[q4 >> 1][(q4 & 1) * 16 + e], v[q4 >> 1][(q4 & 1) * 16 + e + 1]);
                const float m_new =
                    fmaxf(m, fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * c);  // c > 0
                if (m_new != -INFINITY) {
                    const f2 nm = pk(-m_new, -m_new);
                    f2 acc[4] = {pk(0.f, 0.f), pk(0.f, 0.f), pk(0.f, 0.f), pk(0.f, 0.f)};
#pragma unroll
                    for (int ch = 0; ch < 2; ++ch)
#pragma unroll
                        for (int e = 0; e < 32; e += 2) {
                            float x0, x1;
                            upk(fma2(pk(v[ch][e], v[ch][e + 1]), cc, nm), x0, x1);
                            acc[(e >> 1) & 3] = add2(acc[(e >> 1) & 3], pk(ex2(x0), ex2(x1)));
                        }
                    float s0, s1;
                    upk(add2(add2(acc[0], acc[1]), add2(acc[2], acc[3])), s0, s1);
                    l = l * ex2(m - m_new) + (s0 + s1);
                    m = m_new;
                }
            }
            // The pass-A -> pass-B hand-over exchanges the row statistics through
            // named barrier 1.  A warp whose pass-A wait expired records it,
            // arrives at the barrier without waiting and leaves; the others are
            // released and their pass-B waits expire.
            if (!ok) {
                fail(10 + 32 * wg);  // Q K^T in pass A
                named_bar_arrive(1, kSoftThreads);
                break;
            }
            stat[(wg * 2 + 0) * kBM + row] = m;
            stat[(wg * 2 + 1) * kBM + row] = l;
            named_bar_sync(1, kSoftThreads);
            if (kSplit) {
                // this CTA's (max, sum) of every row to every CTA of the cluster
                if (wg == 0) {
                    float mm = stat[row], ll = 0.f;
#pragma unroll
                    for (int g = 1; g < kWG; ++g) mm = fmaxf(mm, stat[g * 2 * kBM + row]);
                    if (mm != -INFINITY)
#pragma unroll
                        for (int g = 0; g < kWG; ++g)
                            ll += stat[(g * 2 + 1) * kBM + row] * ex2(stat[g * 2 * kBM + row] - mm);
                    const uint32_t a = smem_addr(xstat + cluster_ctarank() * kBM + row);
                    for (int q = 0; q < p.split; ++q) st_dsmem_f2(dsmem_addr(a, q), mm, ll);
                }
                cluster_arrive();  // phase 1
                cluster_wait();
                exchanged = true;
            }
            float nl4[4];  // -log2-sum-exp (scaled) of this thread's 4 rows, index 2h + k; -inf for padding rows
            int tq4[4];    // token of each row (T for padding rows)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int rr = quad * 32 + 16 * (i >> 1) + lane / 4 + 8 * (i & 1);
                float mm, ll = 0.f;
                if (kSplit) {  // every CTA adds the ranks in the same order
                    mm = xstat[rr].x;
                    for (int q = 1; q < p.split; ++q) mm = fmaxf(mm, xstat[q * kBM + rr].x);
                    for (int q = 0; q < p.split; ++q) ll += xstat[q * kBM + rr].y * ex2(xstat[q * kBM + rr].x - mm);
                } else {
                    mm = stat[rr];
#pragma unroll
                    for (int g = 1; g < kWG; ++g) mm = fmaxf(mm, stat[g * 2 * kBM + rr]);
#pragma unroll
                    for (int g = 0; g < kWG; ++g)
                        ll += stat[(g * 2 + 1) * kBM + rr] * ex2(stat[g * 2 * kBM + rr] - mm);
                }
                const int gr = x.mt * kBM + rr;
                nl4[i] = gr < rows ? -(mm + __log2f(ll)) : -INFINITY;
                tq4[i] = gr < rows ? gr / G : T;
            }
            // the next unit's Q rows come to L2 during pass B
            prefetch_q(w + wstep);

            // ---------------- pass B: P = exp2(S c - lse) -> TMEM (bf16) and column sums
            // TMEM is read in 16-lane x 256-bit groups: a thread holds 4 rows
            // (quadrant rows 16h + t/4 + 8k, h, k in {0, 1}) x 16 columns
            // (8r + 2(t%4) + e).  P overwrites the first half of the step's own
            // score columns.
            float* part = p.partials ? p.partials + ((static_cast<size_t>(x.u) * p.Hkv + x.hkv) * p.MT + x.mt) * p.P
                                     : nullptr;
            site = 12;
            const int sB = (wg + kWG - (gb + x.ns) % kWG) % kWG;
            b = bar.plus(x.ns + sB);
            for (int s = sB; s < x.ns; s += kWG) {
                const int pb = pbb + s;
                ok = wait_warp(bar0 + kBarSFull + 8 * b.at, b.ph, deadline);
                if (!ok) break;
                tc_fence_after();
                const uint32_t tSb = tSw + (b.at >= kBufs ? b.at - kBufs : b.at) * kStep;
                b.step(kWG);
                float v[2][32];
#pragma unroll
                for (int h = 0; h < 2; ++h) tmem_ld_16x256b_x8(tSb + ((16u * h) << 16), v[h]);
                tmem_ld_wait();
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int r = 0; r < 8; ++r)
#pragma unroll
                        for (int k2 = 0; k2 < 2; ++k2) {
                            const int i = 4 * r + 2 * k2;
                            const float nk = nl4[2 * h + k2];
                            float x0, x1;
                            upk(fma2(pk(v[h][i], v[h][i + 1]), cc, pk(nk, nk)), x0, x1);
                            v[h][i] = ex2(x0);
                            v[h][i + 1] = ex2(x1);
                        }
                const int sg = s + x.s0;
                if (sg >= 2 * x.nfull) {  // a ragged or frame step: keys at or past a row's limit get zero weight
                    int lim4[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        lim4[i] = sg < x.nss ? x.count - sg * kStep
                                             : (p.causal ? min(T, tq4[i] + 1) : T) - (sg - x.nss) * kStep;
                    const int lmin = min(min(lim4[0], lim4[1]), min(lim4[2], lim4[3]));
                    if (lmin < kStep) {
#pragma unroll
                        for (int h = 0; h < 2; ++h)
#pragma unroll
                            for (int r = 0; r < 8; ++r)
#pragma unroll
                                for (int k2 = 0; k2 < 2; ++k2) {
                                    const int i = 4 * r + 2 * k2;
                                    const int col = 8 * r + cq, lim = lim4[2 * h + k2];
                                    v[h][i] = col < lim ? v[h][i] : 0.f;
                                    v[h][i + 1] = col + 1 < lim ? v[h][i + 1] : 0.f;
                                }
                    }
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t pw[16];  // register 2r + k: row k, P column 4r + t%4
#pragma unroll
                    for (int r = 0; r < 8; ++r)
#pragma unroll
                        for (int k2 = 0; k2 < 2; ++k2)
                            pw[2 * r + k2] = pack_bf16x2(v[h][4 * r + 2 * k2], v[h][4 * r + 2 * k2 + 1]);
                    tmem_st_16x128b_x8(tSb + ((16u * h) << 16), pw);
                }
                tmem_st_wait();
                tc_fence_before();
                arrive_at(bar0 + kBarPFull + 8 * (pb & 7));
                // the column sums run while the tensor core does this step's P V:
                // value 2r + e is column 8r + cq + e summed over the thread's rows, then
                // over the 8 lanes that share its columns; the reducer warp adds the warps
                if (part != nullptr) {
                    float cs[16];
#pragma unroll
                    for (int r = 0; r < 8; ++r) {
                        const f2 a = add2(pk(v[0][4 * r], v[0][4 * r + 1]), pk(v[0][4 * r + 2], v[0][4 * r + 3]));
                        const f2 bb = add2(pk(v[1][4 * r], v[1][4 * r + 1]), pk(v[1][4 * r + 2], v[1][4 * r + 3]));
                        upk(add2(a, bb), cs[2 * r], cs[2 * r + 1]);
                    }
                    const float2 sum = lane8_reduce_scatter(cs, lane);  // columns 8 (lane / 4) + cq + {0, 1}
                    if (pb >= 4)  // the reducer has read the step that had the area before
                        ok = wait_warp(bar0 + kBarStageFree + 8 * (pb & 3), ((pb >> 2) & 1) ^ 1, deadline);
                    if (!ok) break;
                    mystage[(pb & 3) * 128] = sum;
                    arrive_at(bar0 + kBarStageFull + 8 * (pb & 3));
                }
            }
            if (!ok) break;
            load_q(w + wstep);  // while the last P V run
            // Frame keys no row of this tile can see receive zero importance here.
            if (part != nullptr && (!kSplit || cluster_ctarank() == 0))
                for (int t = x.nfs * kStep + (threadIdx.x - 128); t < T; t += kSoftThreads) part[B + t] = 0.f;
            // every P V of the unit has completed: O is final, and TMEM's Q and
            // score columns are free for the next unit
            site = 14;
            ok = wait_warp(bar0 + kBarOFull, k & 1, deadline);
            if (!ok) break;
            tc_fence_after();
            prev = x;
            gb += 2 * x.ns;
            pbb += x.ns;
            bar = bar.plus(2 * x.ns);
        }
        if (kSplit) {
            __syncwarp();
            if (!exchanged) {
                cluster_arrive();  // phase 1
                cluster_wait();
            }
            // this CTA's O (fp32; zero if it had no keys) over the idle ring, thread = row
            float* ost = reinterpret_cast<float*>(sSlot);
            if (ok && wg * kOc < D)
#pragma unroll
                for (int c2 = 0; c2 < kOc / 32; ++c2) {
                    const int col = wg * kOc + c2 * 32;
                    float o[32];
                    if (prev.ns > 0) {
                        tmem_ld32(tbase + lane_off + kColO + col, o);
                        tmem_ld_wait();
                    } else {
#pragma unroll
                        for (int e = 0; e < 32; ++e) o[e] = 0.f;
                    }
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        *reinterpret_cast<float4*>(ost + row * L::kOStageLd + col + 4 * e) =
                            make_float4(o[4 * e], o[4 * e + 1], o[4 * e + 2], o[4 * e + 3]);
                }
            __syncwarp();
            cluster_sync();  // phase 2
            if (ok && p.out != nullptr) {  // (the watchdog self-test has no output)
                const int rank = static_cast<int>(cluster_ctarank());
                const int r0 = kBM * rank / p.split, r1 = kBM * (rank + 1) / p.split;
                const uint32_t a0 = smem_addr(ost);
                for (int i = threadIdx.x - 128; i < (r1 - r0) * (D / 4); i += kSoftThreads) {
                    const int rr = r0 + i / (D / 4), c4 = 4 * (i % (D / 4)), my_r = prev.mt * kBM + rr;
                    const uint32_t a = a0 + static_cast<uint32_t>(rr * L::kOStageLd + c4) * 4u;
                    float4 v[kMaxSplit];
#pragma unroll
                    for (int q = 0; q < kMaxSplit; ++q)
                        if (q < p.split) v[q] = ld_dsmem_f4(dsmem_addr(a, q));
#pragma unroll
                    for (int q = 1; q < kMaxSplit; ++q)
                        if (q < p.split) {
                            v[0].x += v[q].x;
                            v[0].y += v[q].y;
                            v[0].z += v[q].z;
                            v[0].w += v[q].w;
                        }
                    if (my_r < rows) {
                        const int t = my_r / G, g = my_r - t * G;
                        *reinterpret_cast<uint2*>(
                            p.out + ((static_cast<size_t>(prev.u) * T + t) * p.Hq + prev.hkv * G + g) * D + c4) =
                            make_uint2(pack_bf16x2(v[0].x, v[0].y), pack_bf16x2(v[0].z, v[0].w));
                    }
                }
            }
            __syncwarp();
            cluster_sync();  // phase 3
        } else if (ok && k >= 1) {
            store_o(prev);  // the last unit's O
        }
        if (!ok) fail(site + 32 * wg);
        tc_fence_before();
        __syncthreads();
    }
}

// The register split must fit the registers the CTA is launched with, or
// setmaxnreg.inc would wait forever.
constexpr int kLaunchRegs = 128;
static_assert(128 * kAuxRegs + kSoftThreads * kSoftRegs <= kThreads * kLaunchRegs, "register split");

// SMs of each device, read by attn_prepare with that device current; the
// persistent grid of a launch is sized for the device current at the launch.
constexpr int kMaxDevices = 64;
int g_num_sms[kMaxDevices] = {};

int current_device_sms()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 1;
    return g_num_sms[dev] > 0 ? g_num_sms[dev] : 1;
}

// Clusters of each size that a device holds at once with the split form's shared
// memory, measured by attn_prepare (0: not measured, or none).
int g_attn_clusters[kMaxDevices][2][kMaxSplit + 1] = {};

// attr: two entries
template <int D>
cudaLaunchConfig_t launch_config(int grid, int S, cudaStream_t st, cudaLaunchAttribute* attr)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = AttnLayout<D>::kAlloc;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = S;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = S > 1 ? 2 : 1;
    return cfg;
}

template <int D, bool kSplit>
cudaError_t prepare_form()
{
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, frame_attn_lse_importance<D, kSplit>);
    if (e != cudaSuccess) return e;
    if (fa.numRegs < kLaunchRegs) return cudaErrorInvalidConfiguration;
    return cudaFuncSetAttribute(frame_attn_lse_importance<D, kSplit>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                AttnLayout<D>::kAlloc);
}

template <int D>
cudaError_t prepare_one()
{
    int dev = 0, sms = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    if ((e = prepare_form<D, false>()) != cudaSuccess || (e = prepare_form<D, true>()) != cudaSuccess) return e;
    for (int S = 2; S <= kMaxSplit; ++S) {
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = launch_config<D>(S, S, nullptr, attr);
        cfg.attrs = attr + 1;  // the cluster size alone
        cfg.numAttrs = 1;
        int n = 0;
        if ((e = cudaOccupancyMaxActiveClusters(&n, frame_attn_lse_importance<D, true>, &cfg)) != cudaSuccess)
            return e;
        g_attn_clusters[dev][D == 128][S] = n;
    }
    g_num_sms[dev] = sms;
    return cudaSuccess;
}

// CTAs per unit: as many as let every unit's cluster be resident at once (so the
// split form runs where the units leave half of the SMs idle or more), if each CTA
// then has kMinSaved tiles fewer than the unit: the two exchanges cost ~4.4 us, a
// tile 0.8.  Per launch (ncu): 7 tiles whole ~17 us, on two CTAs 21.5; 15 tiles
// whole 23.5 us, on three 20.
constexpr int kMinSaved = 7;
template <int D>
int split_for(long long W, int tiles)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 1;
    for (int S = kMaxSplit; S >= 2; --S)
        if (W <= g_attn_clusters[dev][D == 128][S] && tiles - (tiles + S - 1) / S >= kMinSaved) return S;
    return 1;
}

// One CTA per SM (at most one per work unit), each walking its units in order; or
// a cluster per unit.
template <int D>
cudaError_t launch_one(const CUtensorMap& tm_sk, const CUtensorMap& tm_sv, const CUtensorMap& tm_fk,
                       const CUtensorMap& tm_fv, const AttnParams& p0, int U, cudaStream_t st)
{
    AttnParams p = p0;
    p.U = U;
    const long long W = static_cast<long long>(p.MT) * p.Hkv * U;
    if (W <= 0) return cudaSuccess;
    if (W > 0x7FFFFFFFll) return cudaErrorInvalidValue;
    p.split = split_for<D>(W, (p.keys_hint + kBN - 1) / kBN + (p.T + kBN - 1) / kBN);
    const int sms = current_device_sms();
    const int grid = p.split > 1 ? static_cast<int>(W) * p.split : static_cast<int>(W < sms ? W : sms);
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = launch_config<D>(grid, p.split, st, attr);
    return p.split > 1 ? cudaLaunchKernelEx(&cfg, frame_attn_lse_importance<D, true>, tm_sk, tm_sv, tm_fk, tm_fv, p)
                       : cudaLaunchKernelEx(&cfg, frame_attn_lse_importance<D, false>, tm_sk, tm_sv, tm_fk, tm_fv, p);
}

}  // namespace

int device_sm_count() { return current_device_sms(); }

size_t attn_smem_bytes(int D)
{
    return D == 64 ? AttnLayout<64>::kAlloc : AttnLayout<128>::kAlloc;
}

cudaError_t attn_prepare(int D)
{
    return D == 64 ? prepare_one<64>() : prepare_one<128>();
}

cudaError_t launch_attn(int D, const CUtensorMap& tm_sk, const CUtensorMap& tm_sv,
                        const CUtensorMap& tm_fk, const CUtensorMap& tm_fv, const AttnParams& p,
                        int U, cudaStream_t st)
{
    const cudaError_t e = D == 64 ? launch_one<64>(tm_sk, tm_sv, tm_fk, tm_fv, p, U, st)
                                  : launch_one<128>(tm_sk, tm_sv, tm_fk, tm_fv, p, U, st);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace statekv
