// Exact top-k of a row held in registers, by a histogram over the keys' own
// range and a ranking of the bucket that holds the k-th key.
//
// A block of NT threads owns a row of up to NT * KPT positions: value i of a
// thread is position warp * 32 * KPT + (i / 4) * 128 + lane * 4 + i % 4, so a
// warp's loads of four consecutive positions per lane are coalesced.  Keys are
// order-preserving uint32 (larger is better), 0 marks an ineligible position;
// ties go to the lower position.
//
// The 4096 buckets divide the range from the smallest to the largest eligible
// key: the scores of a row lie within a few octaves, most of them within one, so
// their bits above the range say nothing and few of them share a bucket (neither
// its shared-memory counter).  The bucket of the k-th key then holds some ten
// keys, which are compacted and ranked against each other at once: five block
// barriers in all, where an MSB radix select takes one per 4-bit digit and a
// sweep of the row for most of them.  A bucket that is too large is divided into
// 4096 again, and equal keys are taken by position.
#pragma once

#include "kvec_internal.cuh"

namespace kvec {

constexpr int kSelBits = 12;
constexpr int kSelBins = 1 << kSelBits;
constexpr int kSelList = 128;    // entries of the k-th key's bucket that are ranked directly

struct HistSelectShared {
    uint32_t hist[kSelBins];                  // zero between selections
    unsigned long long list[kSelList];        // key << 32 | ~position
    int wsum[32];
    uint32_t wmin[32], wmax[32];
    int bin, above, count, fill;
};

template <int NT, int KPT>
struct HistSelect {
    static_assert(KPT == 16 || KPT == 32, "four positions per group of a thread's values");
    static_assert(NT >= kSelList && NT * 4 <= kSelBins, "an entry and four bins per thread");
    static constexpr int kPositions = NT * KPT;
    static constexpr int kWords = kPositions / 32;
    static constexpr int kBPT = kSelBins / NT;   // bins per thread
    static constexpr int kWarps = NT / 32;

    HistSelectShared& sm;
    int k;          // keys to select
    int kk = 0;     // of them, in the threshold bucket
    int m = 0;      // keys in the threshold bucket

    __device__ __forceinline__ static int position(int i) {
        return (int)(threadIdx.x >> 5) * 32 * KPT + (i >> 2) * 128 + (int)(threadIdx.x & 31) * 4 + (i & 3);
    }

    // Once per kernel, before a block barrier that precedes the first selection.
    __device__ __forceinline__ static void clear(HistSelectShared& sm) {
        for (int i = threadIdx.x; i < kSelBins; i += NT) sm.hist[i] = 0u;
    }

    // The values above the threshold bucket (bit i: value i), and in `match` those
    // inside it, of which finish() takes the best.  k >= 1 and at least k keys
    // are eligible.
    __device__ __forceinline__ uint32_t begin(const uint32_t (&key)[KPT], uint32_t& match) {
        const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
        uint32_t kmin = 0xffffffffu, kmax = 0u, active = 0u;
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
            kmin = min(kmin, key[i] - 1u);   // an ineligible key wraps to the top
            kmax = max(kmax, key[i]);
            active |= (key[i] != 0u ? 1u : 0u) << i;
        }
        kmin = __reduce_min_sync(0xffffffffu, kmin);
        kmax = __reduce_max_sync(0xffffffffu, kmax);
        if (lane == 0) {
            sm.wmin[warp] = kmin;
            sm.wmax[warp] = kmax;
        }
        if (tid == 0) sm.fill = 0;
        __syncthreads();
        uint32_t lo = __reduce_min_sync(0xffffffffu, lane < kWarps ? sm.wmin[lane] : 0xffffffffu) + 1u;
        const uint32_t range = __reduce_max_sync(0xffffffffu, lane < kWarps ? sm.wmax[lane] : 0u) - lo;
        int shift = max(32 - kSelBits - __clz(range), 0);   // range >> shift < kSelBins
        uint32_t sure = 0u;
        kk = k;
        for (;;) {
#pragma unroll
            for (int i = 0; i < KPT; ++i)
                if ((active >> i) & 1u) atomicAdd(&sm.hist[(key[i] - lo) >> shift], 1u);
            __syncthreads();
            // Thread t sums the bins 4095 - kBPT t and the kBPT - 1 below, clears them,
            // and the thread whose sums straddle kk finds the bin.
            uint32_t c[kBPT];
            int own = 0;
#pragma unroll
            for (int b = 0; b < kBPT; b += 4) {
                uint4* src = reinterpret_cast<uint4*>(&sm.hist[kSelBins - kBPT * (tid + 1) + kBPT - 4 - b]);
                const uint4 v = *src;
                *src = make_uint4(0u, 0u, 0u, 0u);
                c[b] = v.w;
                c[b + 1] = v.z;
                c[b + 2] = v.y;
                c[b + 3] = v.x;
                own += (int)(v.x + v.y + v.z + v.w);
            }
            int incl = own;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (lane == 31) sm.wsum[warp] = incl;
            __syncthreads();
            int before = lane < kWarps && lane < warp ? sm.wsum[lane] : 0;
            before = __reduce_add_sync(0xffffffffu, before) + incl - own;
            if (before < kk && kk <= before + own) {
                int at = before;
#pragma unroll
                for (int b = 0; b < kBPT; ++b) {
                    if (at < kk && kk <= at + (int)c[b]) {
                        sm.bin = kSelBins - 1 - (kBPT * tid + b);
                        sm.above = at;
                        sm.count = (int)c[b];
                    }
                    at += (int)c[b];
                }
            }
            __syncthreads();
            kk -= sm.above;
            m = sm.count;
            // The bucket holds the keys [first, first + 2^shift).
            const uint32_t first = lo + ((uint32_t)sm.bin << shift), width = 1u << shift;
            match = 0u;
            uint32_t over = 0u;
#pragma unroll
            for (int i = 0; i < KPT; ++i) {
                const uint32_t d = key[i] - first;   // wraps below the bucket
                if (d < width) match |= 1u << i;
                if (key[i] >= first) over |= 1u << i;
            }
            match &= active;
            sure |= over & active & ~match;
            if (m == kk) {   // the bucket is taken whole
                sure |= match;
                match = 0u;
            }
            if (m == kk || m <= kSelList || shift == 0) return sure;
            active = match;
            lo = first;
            shift = max(shift - kSelBits, 0);
        }
    }

    // ORs the best kk of the bucket into bits[] (one bit per position, shared
    // memory).  Every store of begin()'s positions into bits[] precedes it in
    // program order; the bits are complete after the next barrier.
    __device__ __forceinline__ void finish(const uint32_t (&key)[KPT], uint32_t match, uint32_t* bits) {
        const int tid = threadIdx.x, lane = tid & 31;
        if (m == kk) return;   // the same for the whole block
        if (m <= kSelList) {
            const int c = __popc(match);
            if (__any_sync(0xffffffffu, c != 0)) {
                int incl = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += y;
                }
                int at = 0;
                if (lane == 31) at = atomicAdd(&sm.fill, incl);
                at = __shfl_sync(0xffffffffu, at, 31) + incl - c;
#pragma unroll
                for (int i = 0; i < KPT; ++i)
                    if ((match >> i) & 1u)
                        sm.list[at++] = ((unsigned long long)key[i] << 32) | (uint32_t)~(uint32_t)position(i);
            }
            __syncthreads();
            // Threads per entry: a power of two, at most a warp's.
            int per = 1;
            while (per < 32 && per * 2 * m <= NT) per *= 2;
            const int sub = tid & (per - 1), e = tid / per;   // NT >= kSelList: an entry for every `per` threads
            if (e - lane / per < m) {   // whole warps stay together
                const unsigned long long mine = e < m ? sm.list[e] : 0ull;
                int rank = 0;
                for (int j = sub; j < m; j += per) rank += sm.list[j] > mine ? 1 : 0;
                for (int o = 1; o < per; o <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
                if (sub == 0 && e < m && rank < kk) {
                    const uint32_t pos = ~(uint32_t)mine;
                    atomicOr(&bits[pos >> 5], 1u << (pos & 31));
                }
            }
            return;
        }
        store_or(lowest(sm, match, kk), bits);
    }

    // The `take` lowest positions of the block's values in `match`.  Before a
    // thread's: earlier warps, earlier groups of this warp, lower lanes, lower
    // values of the group.
    __device__ __forceinline__ static uint32_t lowest(HistSelectShared& sm, uint32_t match, int take) {
        const int tid = threadIdx.x, lane = tid & 31;
        const int wt = __reduce_add_sync(0xffffffffu, __popc(match));
        if (lane == 0) sm.wsum[tid >> 5] = wt;
        __syncthreads();
        int before = lane < (tid >> 5) ? sm.wsum[lane] : 0;
        before = __reduce_add_sync(0xffffffffu, before);
        uint32_t taken = 0u;
#pragma unroll
        for (int g = 0; g < KPT / 4; ++g) {
            const int c = __popc((match >> (4 * g)) & 15u);
            int incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            int rank = before + incl - c;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const uint32_t bit = 1u << (4 * g + e);
                if (match & bit) {
                    if (rank < take) taken |= bit;
                    ++rank;
                }
            }
            before += __shfl_sync(0xffffffffu, incl, 31);
        }
        return taken;
    }

    // bits[] gets the values of `sel` as plain stores: every byte of the row's
    // words is written (lanes 2 j and 2 j + 1 hold a byte's nibbles).
    __device__ __forceinline__ static void store(uint32_t sel, uint32_t* bits) {
        uint8_t* bytes = reinterpret_cast<uint8_t*>(bits);
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int g = 0; g < KPT / 4; ++g) {
            const uint32_t nib = (sel >> (4 * g)) & 15u;
            const uint32_t hi = __shfl_down_sync(0xffffffffu, nib, 1);
            if ((lane & 1) == 0) bytes[position(4 * g) >> 3] = (uint8_t)(nib | (hi << 4));
        }
    }
    __device__ __forceinline__ static void store_or(uint32_t sel, uint32_t* bits) {
#pragma unroll
        for (int g = 0; g < KPT / 4; ++g) {
            const uint32_t nib = (sel >> (4 * g)) & 15u;
            const int pos = position(4 * g);
            if (nib) atomicOr(&bits[pos >> 5], nib << (pos & 31));
        }
    }
};

}  // namespace kvec
