// How the decode-cache append inside the selection's launch numbers its copies.
// Plain C++: a host program can check it.
#pragma once

#ifdef __CUDACC__
#define SKV_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define SKV_HOST_DEVICE inline
#endif

namespace statekv {

constexpr int kSelThreads = 640;
constexpr int kAppendBatch = 8;  // copies per thread in flight

// Copies of one matrix (K or V) of one unit, 16 bytes each, in source order
// [token][KV head][chunk]; a unit's copies are K's, then V's.
SKV_HOST_DEVICE long long append_copies(int T, int Hkv, int D) { return static_cast<long long>(T) * Hkv * (D / 8); }

// Indexes are 32-bit where every index formed (the last copy plus a round of all
// CTAs' batches) fits, 64-bit from 2^30 copies on: 4096 tokens of 16,384 heads of
// 128 are 2^31, and the configuration allows 65,535 heads.
SKV_HOST_DEVICE bool append_narrow(int T, int Hkv, int D) { return 2 * append_copies(T, Hkv, D) <= 1ll << 30; }

// Append CTAs per unit: one batch of copies for each thread, up to eight CTAs, and
// whole clusters where the heads' CTAs come in clusters of `split` (1, 2, 4 or 8).
inline int append_ctas(int T, int Hkv, int D, int split)
{
    const long long per_cta = kAppendBatch * kSelThreads;
    const long long n = (2 * append_copies(T, Hkv, D) + per_cta - 1) / per_cta;
    return (static_cast<int>(n < 8 ? n : 8) + split - 1) / split * split;
}

struct AppendAt {
    int t, hkv, ch;
};

// Token, KV head and chunk of copy i < 2 per.
template <class I>
SKV_HOST_DEVICE AppendAt append_at(I i, I per, int Hkv, int chunks)
{
    const I r = i < per ? i : i - per;
    const int t = static_cast<int>(r / (Hkv * chunks)), hc = static_cast<int>(r - static_cast<I>(t) * (Hkv * chunks));
    return {t, hc / chunks, hc % chunks};
}

}  // namespace statekv
