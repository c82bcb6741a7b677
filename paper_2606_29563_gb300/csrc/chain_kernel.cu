// Section 4.2 over a run of consecutive layers: P' = P + lambda * I * (1 - n_t /
// (l + 1)), the preserved tokens stay, the rest of B - w goes to the largest P',
// the last w tokens are kept, and the layer's union moves the coverage counts.
//
// Only this step is serial across layers, so one launch walks all the layers
// whose scores are ready.  A cluster of Hkv CTAs serves a sequence, a CTA per KV
// head: every thread keeps the counts n_t of its positions (in shared memory for
// the longest rows), builds their keys in registers, and the heads' kept bits meet
// over distributed shared memory behind one cluster barrier per layer, while the
// next layer's scores are being copied in.  A chain of dependent steps (a histogram
// between five block barriers, then the cluster's) bounds a layer, not bandwidth.
// Per-layer launches instead pass the union and the counts through L2 and stage the
// keys in shared memory: 14 to 17 us per layer of one 8192-token sequence where this
// takes about 5.5.
#include <cooperative_groups.h>

#include "hist_select.cuh"
#include "sm100_ptx.cuh"

namespace kvec {

namespace {

namespace cg = cooperative_groups;

// Rows of up to 16384 positions have their importances in shared memory beside the
// scores; longer ones, whose threads need the registers, their counts.
__host__ __device__ constexpr bool chain_stages_i(int nt, int kpt) { return nt * kpt <= 16384; }
__host__ __device__ constexpr int chain_smem_bytes(int nt, int kpt) {
    return nt * kpt * (int)sizeof(float) + nt * kpt * (chain_stages_i(nt, kpt) ? (int)sizeof(float) : 1);
}

__device__ __forceinline__ void copy_async_word(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(ptx::smem_u32(dst)), "l"(src) : "memory");
}

struct ChainArgs {
    Geometry G;
    const int* cu;
    uint8_t* state;
    int* refused;      // [batch] 1: the call would take this state past 255 layers (set by its first launch)
    int* err;
    int l0, nl, ncall; // layers [l0, l0 + nl) of a call of ncall
    Slot sl[kMaxGroup];
};

// What the CTAs of a cluster read from each other in a joint selection.
struct JointShared {
    uint32_t kmin, kmax;
    int total;                            // keys in this CTA's slice of the buckets
    int bin, above, count;                // the bucket of the k-th key, in the CTA whose slice holds it
    int fill;                             // list entries, or equal keys
    unsigned long long list[kSelList];    // this head's keys in that bucket: key << 32 | ~(head, position)
};

// The k largest of the keys in `active` over every CTA of the cluster (a KV head
// each), ORed into their heads' bits; ties go to the lower head, then to the lower
// position.  HistSelect's buckets, over the cluster's range of keys: each CTA
// counts its own keys, CTA r adds up the r-th slice of the buckets from the top,
// and the one whose slice holds the k-th key names its bucket.  At least k keys
// are active.  The bits are complete after the next block barrier.
template <int NT, int KPT>
__device__ __noinline__ void joint_select(const uint32_t* keys, uint32_t active, int k, HistSelectShared& sm,
                                          JointShared& js, uint32_t* bits) {
    using HS = HistSelect<NT, KPT>;
    cg::cluster_group cluster = cg::this_cluster();
    const int nc = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t key[KPT];
    uint32_t kmin = 0xffffffffu, kmax = 0u;
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
        key[i] = keys[i];
        if ((active >> i) & 1u) {
            kmin = min(kmin, key[i]);
            kmax = max(kmax, key[i]);
        }
    }
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0) {
        sm.wmin[warp] = kmin;
        sm.wmax[warp] = kmax;
    }
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < HS::kWarps; ++w) {
            kmin = min(kmin, sm.wmin[w]);
            kmax = max(kmax, sm.wmax[w]);
        }
        js.kmin = kmin;
        js.kmax = kmax;
        js.fill = 0;
    }
    cluster.sync();
    uint32_t lo = 0xffffffffu, hi = 0u;
    if (lane < nc) {
        lo = *cluster.map_shared_rank(&js.kmin, lane);
        hi = *cluster.map_shared_rank(&js.kmax, lane);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    int shift = max(32 - kSelBits - __clz(hi - lo), 0);
    const int slice = (kSelBins + nc - 1) / nc, per = (slice + NT - 1) / NT;   // buckets of a CTA, of a thread
    uint32_t sure = 0u, match = 0u;
    int kk = k, m = 0;
    for (;;) {
#pragma unroll
        for (int i = 0; i < KPT; ++i)
            if ((active >> i) & 1u) atomicAdd(&sm.hist[(key[i] - lo) >> shift], 1u);
        cluster.sync();
        // Buckets from the top: this CTA's slice, this thread's `per` of it.
        int own = 0;
        for (int b = 0; b < per; ++b) {
            const int i = tid * per + b, bin = kSelBins - 1 - (rank * slice + i);
            if (i >= slice || bin < 0) break;
            for (int r = 0; r < nc; ++r) own += (int)*cluster.map_shared_rank(&sm.hist[bin], r);
        }
        int incl = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) sm.wsum[warp] = incl;
        __syncthreads();
        const int ws = lane < HS::kWarps ? sm.wsum[lane] : 0;
        const int total = __reduce_add_sync(0xffffffffu, ws);
        int before = __reduce_add_sync(0xffffffffu, lane < warp ? ws : 0) + incl - own;
        if (tid == 0) js.total = total;
        cluster.sync();
        int owner = 0, above = 0;   // the CTA whose slice holds the kk-th key, and the keys in the slices above it
        for (; owner + 1 < nc; ++owner) {
            const int t = *cluster.map_shared_rank(&js.total, owner);
            if (kk <= above + t) break;
            above += t;
        }
        if (owner == rank && above + before < kk && kk <= above + before + own) {
            int at = above + before;
            for (int b = 0; b < per; ++b) {
                const int bin = kSelBins - 1 - (rank * slice + tid * per + b);
                if (tid * per + b >= slice || bin < 0) break;
                int c = 0;
                for (int r = 0; r < nc; ++r) c += (int)*cluster.map_shared_rank(&sm.hist[bin], r);
                if (at < kk && kk <= at + c) {
                    js.bin = bin;
                    js.above = at;
                    js.count = c;
                }
                at += c;
            }
        }
        cluster.sync();
        HS::clear(sm);   // every count has been read
        const uint32_t bin = (uint32_t)*cluster.map_shared_rank(&js.bin, owner);
        kk -= *cluster.map_shared_rank(&js.above, owner);
        m = *cluster.map_shared_rank(&js.count, owner);
        match = 0u;
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
            const uint32_t on = (active >> i) & 1u, d = (key[i] - lo) >> shift;
            sure |= (on & (d > bin ? 1u : 0u)) << i;
            match |= (on & (d == bin ? 1u : 0u)) << i;
        }
        if (m == kk || m <= kSelList || shift == 0) break;
        active = match;
        lo += bin << shift;
        shift = max(shift - kSelBits, 0);
        __syncthreads();   // the counters are clear
    }
    if (m == kk) {   // the bucket is taken whole
        HS::store_or(sure | match, bits);
        return;
    }
    HS::store_or(sure, bits);
    if (m <= kSelList) {
        // The heads' entries of the bucket side by side, ranked against each other.
#pragma unroll
        for (int i = 0; i < KPT; ++i)
            if ((match >> i) & 1u)
                js.list[atomicAdd(&js.fill, 1)] =
                    ((unsigned long long)key[i] << 32) | (uint32_t)~(((uint32_t)rank << 24) | (uint32_t)HS::position(i));
        cluster.sync();
        int at = 0;
        for (int r = 0; r < nc; ++r) {
            const int n = *cluster.map_shared_rank(&js.fill, r);
            for (int e = tid; e < n; e += NT) sm.list[at + e] = *cluster.map_shared_rank(&js.list[e], r);
            at += n;
        }
        __syncthreads();
        if (tid < m) {
            const unsigned long long mine = sm.list[tid];
            const uint32_t where = ~(uint32_t)mine;
            if ((int)(where >> 24) == rank) {
                int better = 0;
                for (int j = 0; j < m; ++j) better += sm.list[j] > mine ? 1 : 0;
                const uint32_t pos = where & 0xffffffu;
                if (better < kk) atomicOr(&bits[pos >> 5], 1u << (pos & 31));
            }
        }
        return;
    }
    // More than kSelList equal keys: the lower heads', then the lower positions'.
    const int c = __reduce_add_sync(0xffffffffu, __popc(match));
    if (lane == 0 && c) atomicAdd(&js.fill, c);
    cluster.sync();
    for (int r = 0; r < rank; ++r) kk -= *cluster.map_shared_rank(&js.fill, r);
    HS::store_or(HS::lowest(sm, match, max(kk, 0)), bits);
}

template <int NT, int KPT, bool ADA>
__global__ void __launch_bounds__(NT, 1) chain_kernel(const __grid_constant__ ChainArgs A) {
    using HS = HistSelect<NT, KPT>;
    __shared__ HistSelectShared sm;
    __shared__ __align__(16) uint32_t bits[2][HS::kWords];   // this head's kept positions, by layer parity
    __shared__ __align__(16) uint32_t uni[HS::kWords];       // the last layer's union
    __shared__ uint32_t spres[HS::kWords];                   // the layer's preserved bits
    __shared__ JointShared js[1];
    __shared__ uint64_t staged;   // the layer's scores (and importances) are there
    // The layer's scores by position, then its importances, or the counts as [KPT / 4][NT]
    // words of four.
    extern __shared__ __align__(128) float4 sP[];
    constexpr bool kStageI = chain_stages_i(NT, KPT);
    float4* const sI = sP + NT * KPT / 4;
    uint32_t* const sN = reinterpret_cast<uint32_t*>(sI);
    cg::cluster_group cluster = cg::this_cluster();
    const int h = (int)cluster.block_rank(), s = blockIdx.y;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    HS::clear(sm);
    if (tid == 0) {
        ptx::mbar_init(&staged, 1);
        ptx::fence_barrier_init();
    }
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    const int Hkv = A.G.Hkv, words = A.G.words, budget = A.G.budget;
    const int L = __ldg(&A.cu[s + 1]) - __ldg(&A.cu[s]);
    const int Lc = L - A.G.wk;
    const int wordsL = (L + 31) >> 5;
    const bool select = L > budget;
    const size_t row = (size_t)s * Hkv + h;
    uint8_t* st = A.state + (size_t)s * A.G.state_stride;
    uint8_t* nst = st + A.G.state_n_off;
    const uint32_t ell0 = __ldcg(reinterpret_cast<const uint32_t*>(st));   // layers before this launch
    // n_t is 8-bit: a state may count at most 255 layers.  Every launch of a
    // refused call leaves the state as it was.
    const bool refuse = A.l0 == 0 ? ell0 + (uint32_t)A.ncall > 255u : __ldcg(&A.refused[s]) != 0;
    if (A.l0 == 0 && h == 0 && tid == 0) A.refused[s] = refuse ? 1 : 0;
    if (refuse) {   // the same for the whole cluster
        // What follows on the stream waits for this grid alone, which so waits too.
        asm volatile("griddepcontrol.wait;\n" ::: "memory");
        if (tid == 0) atomicExch(A.err, 2);
        return;
    }
    uint32_t n4[kStageI ? KPT / 4 : 1];   // counts of this thread's positions, four bytes a word
    auto counts = [&](int g) -> uint32_t& {
        if constexpr (kStageI) return n4[g];
        return sN[g * NT + tid];
    };
#pragma unroll
    for (int g = 0; g < KPT / 4; ++g) {
        const int t = HS::position(4 * g);
        counts(g) = t < L ? __ldcg(reinterpret_cast<const uint32_t*>(nst + t)) : 0u;
    }
    // The state is the previous call's, complete before this call's first kernel began;
    // the scores come from the kernels before this one.
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    uint32_t top = 0u;   // bit l: the head takes O' in layer l
    for (int l = 0; l < A.nl; ++l) top |= (__ldg(&A.sl[l].htop[row]) != 0 ? 1u : 0u) << l;
    // A layer's scores P and importance I come by bulk copies into shared memory, issued
    // once the layer before has its keys: beside the score and window grids an L2 round
    // trip takes 2 us and more.  (Bulk, since cp.async by every thread kept it from its
    // own work: 32 layers of 8192 tokens 403 -> 390 us, 28 of the Qwen shape at 16384
    // 498 -> 477.  Rows of more than 16384 positions leave no room for I, which is read
    // where it is used: 32 layers of 32768 tokens 1086 us; loaded under the cluster
    // barrier into 32 registers of the 64 that 1024 threads have, 1237.)
    auto stage = [&](int l) {
        const Slot& sl = A.sl[l];
        if (tid == 0) {
            const float* P = (((top >> l) & 1u) ? sl.POe : sl.PO) + row * A.G.ML;
            const uint32_t bytes = (uint32_t)((Lc + 3) & ~3) * (uint32_t)sizeof(float);
            ptx::mbar_arrive_expect_tx(&staged, kStageI ? 2 * bytes : bytes);
            ptx::bulk_load(sP, P, bytes, &staged);
            if constexpr (kStageI) ptx::bulk_load(sI, sl.I + (size_t)s * A.G.ML, bytes, &staged);
        }
        if (tid < HS::kWords && tid < wordsL) copy_async_word(&spres[tid], sl.pres + row * words + tid);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    __syncthreads();   // the barrier is set up
    if (select) stage(0);
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    for (int l = 0; l < A.nl; ++l) {
        uint32_t* b = bits[l & 1];
        uint32_t keep = 0u;   // positions kept without ranking: preserved tokens and the kept tail
        if (select) {
            const float inv_l1 = __frcp_rn((float)(ell0 + (uint32_t)l + 1u));
            // P' of the last layer of a call is kept for inspection (kvec_debug_scores).
            float* Pp = A.l0 + l + 1 == A.ncall ? A.sl[l].Pprime + row * A.G.ML : nullptr;
            // A copy that never lands is reported; the call's results are then void.
            if (!ptx::mbar_wait(&staged, l & 1)) atomicExch(A.err, 3);
            uint32_t key[KPT];
#pragma unroll
            for (int g = 0; g < KPT / 4; ++g) {
                const int t0 = HS::position(4 * g);
                const float4 p = t0 < Lc ? sP[t0 >> 2] : make_float4(0.f, 0.f, 0.f, 0.f);
                const uint32_t pres = t0 < Lc ? (spres[t0 >> 5] >> (t0 & 31)) & 15u : 0u;
                // Positions that do not compete: preserved ones, and from Lc on.
                const int lim = Lc - t0;
                const uint32_t out4 = lim >= 4 ? pres : lim > 0 ? pres | (15u << lim) : 15u;
                keep |= pres << (4 * g);
                if (lim < 4 && t0 < L)   // the kept tail [Lc, L)
                    keep |= ((15u << max(lim, 0)) & (t0 + 4 <= L ? 15u : (1u << (L - t0)) - 1u) & 15u) << (4 * g);
                const float p4[4] = {p.x, p.y, p.z, p.w};
                float4 iv;
                if constexpr (kStageI)
                    iv = t0 < Lc ? sI[t0 >> 2] : make_float4(0.f, 0.f, 0.f, 0.f);
                else
                    iv = t0 < Lc ? __ldg(reinterpret_cast<const float4*>(A.sl[l].I + (size_t)s * A.G.ML + t0)) : make_float4(0.f, 0.f, 0.f, 0.f);
                const float i4[4] = {iv.x, iv.y, iv.z, iv.w};
                const uint32_t nc = counts(g);
                float out[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    // coverage = n_t / (l + 1), by the rounded reciprocal; the byte n_t in
                    // the mantissa of 2^23 + n_t gives its float without a conversion.
                    const float n = __uint_as_float(__byte_perm(nc, 0x4b000000u, 0x7650u + e)) - 8388608.f;
                    const float coverage = n * inv_l1;
                    const float pp = p4[e] + A.G.lambda * (i4[e] * (1.f - coverage));
                    out[e] = pp;
                    key[4 * g + e] = (out4 >> e) & 1u ? 0u : float_order_key(pp);
                }
                if (Pp && t0 < Lc) *reinterpret_cast<float4*>(Pp + t0) = make_float4(out[0], out[1], out[2], out[3]);
            }
            if (l + 1 < A.nl) {
                __syncthreads();   // the scores and the preserved bits have been read
                stage(l + 1);
            }
            if (A.G.f0 > 0) {
                HS hs{sm, A.G.f0};
                uint32_t match;
                keep |= hs.begin(key, match);
                HS::store(keep, b);
                hs.finish(key, match, b);
            } else {
                HS::store(keep, b);
            }
            if constexpr (ADA) {
                // Head-wise adaptive fill: the sequence's other extras = Hkv * (k2 - f0)
                // slots go to the best of all heads' remaining candidates.  (Preserved
                // tokens are exactly Kp of the Lc candidates, so there are enough.)
                if (A.G.extras > 0) {
                    __syncthreads();
                    uint32_t rest = 0u;
#pragma unroll
                    for (int i = 0; i < KPT; ++i) {
                        const int t = HS::position(i);
                        rest |= (key[i] != 0u && !((b[t >> 5] >> (t & 31)) & 1u) ? 1u : 0u) << i;
                    }
                    __syncthreads();   // the bits have been read
                    joint_select<NT, KPT>(key, rest, A.G.extras, sm, js[0], b);
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < KPT; ++i) keep |= (HS::position(i) < L ? 1u : 0u) << i;
            HS::store(keep, b);
        }
        // The heads' kept bits: written above, read below by every CTA of the
        // cluster.  A buffer is written again two layers on, after the next
        // barrier, which every reader passes first.
        asm volatile("cp.async.wait_all;\n" ::: "memory");   // the next layer's preserved bits, read by other threads
        cluster.sync();
        // A warp's union words: lane (4 hh + c) takes four words of head hh.
#pragma unroll
        for (int part = 0; part < KPT / 16; ++part) {
            const int w0 = warp * KPT + part * 16;
            const int hh = lane >> 2;
            uint4 u = make_uint4(0u, 0u, 0u, 0u);
            if (hh < Hkv) u = *reinterpret_cast<const uint4*>(cluster.map_shared_rank(&b[w0 + (lane & 3) * 4], hh));
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) {
                u.x |= __shfl_xor_sync(0xffffffffu, u.x, o);
                u.y |= __shfl_xor_sync(0xffffffffu, u.y, o);
                u.z |= __shfl_xor_sync(0xffffffffu, u.z, o);
                u.w |= __shfl_xor_sync(0xffffffffu, u.w, o);
            }
            __syncwarp();   // the last layer's words have been read
            if (lane < 4) *reinterpret_cast<uint4*>(&uni[w0 + lane * 4]) = u;
            __syncwarp();
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                const uint32_t nib = (uni[w0 + g * 4 + (lane >> 3)] >> ((lane & 7) * 4)) & 15u;
                counts(part * 4 + g) += (nib * 0x00204081u) & 0x01010101u;   // a byte per position: no count passes 255
            }
            // The head's kept positions, for the gather.
            if (lane < 16 && w0 + lane < wordsL) A.sl[l].sel[row * words + w0 + lane] = b[w0 + lane];
        }
    }
    // Counts, union and header for the next launch or call; the CTAs take slices
    // of the positions (all counts were read before the first barrier).
    const int fper = (((L + Hkv - 1) / Hkv) + 31) & ~31;
    const int f0 = min(h * fper, L), f1 = min(f0 + fper, L);
#pragma unroll
    for (int g = 0; g < KPT / 4; ++g) {
        const int t = HS::position(4 * g);
        if (t < f0 || t >= f1) continue;
        if (t + 4 <= L) {
            *reinterpret_cast<uint32_t*>(nst + t) = counts(g);
        } else {
            for (int e = 0; t + e < L; ++e) nst[t + e] = (uint8_t)(counts(g) >> (8 * e));
        }
    }
    if (h == 0) {
        uint32_t* last_union = reinterpret_cast<uint32_t*>(st + A.G.state_union_off);
        for (int w = lane; w < KPT; w += 32) {
            const int wd = warp * KPT + w;
            if (wd < words) last_union[wd] = wd < wordsL ? uni[wd] : 0u;
        }
        for (int wd = HS::kWords + tid; wd < words; wd += NT) last_union[wd] = 0u;
        if (tid == 0) {
            reinterpret_cast<uint32_t*>(st)[0] = ell0 + (uint32_t)A.nl;
            reinterpret_cast<uint32_t*>(st)[1] = (uint32_t)L;
        }
    }
    cluster.sync();   // no CTA leaves while another still reads its bits
}

template <int NT, int KPT, bool ADA>
cudaError_t launch_one(const ChainArgs& a, cudaStream_t st, int priority, bool programmatic) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.G.Hkv, a.G.batch);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = chain_smem_bytes(NT, KPT);
    cfg.stream = st;
    cudaLaunchAttribute attr[3];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = a.G.Hkv;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributePriority;
    attr[1].val.priority = priority;
    attr[2].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[2].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = programmatic ? 3 : 2;
    return cudaLaunchKernelEx(&cfg, chain_kernel<NT, KPT, ADA>, a);
}

// As few threads as hold the longest row with 16 values each (32 from 16384 on).  One
// layer of 8192 positions takes longer with 1024 threads and 8 values each (barriers;
// 32 layers 395 against 387 us) and one of 16384 with 512 and 32 (28 layers of the
// Qwen shape 477 against 468).
template <bool ADA>
cudaError_t launch_for(const Geometry& g, const ChainArgs& a, cudaStream_t st, int priority, bool pdl) {
    if (g.max_len <= 256 * 16) return launch_one<256, 16, ADA>(a, st, priority, pdl);
    if (g.max_len <= 512 * 16) return launch_one<512, 16, ADA>(a, st, priority, pdl);
    if (g.max_len <= 1024 * 16) return launch_one<1024, 16, ADA>(a, st, priority, pdl);
    return launch_one<1024, 32, ADA>(a, st, priority, pdl);
}

template <int NT, int KPT>
cudaError_t configure_one() {
    for (auto fn : {chain_kernel<NT, KPT, false>, chain_kernel<NT, KPT, true>}) {
        const cudaError_t e =
            cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, chain_smem_bytes(NT, KPT));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t configure_chain() {
    cudaError_t e = configure_one<256, 16>();
    if (e == cudaSuccess) e = configure_one<512, 16>();
    if (e == cudaSuccess) e = configure_one<1024, 16>();
    if (e == cudaSuccess) e = configure_one<1024, 32>();
    return e;
}

bool chain_fits(const Geometry& g) { return g.Hkv <= kMaxClusterHeads && g.max_len <= kMaxRegisterRow; }

cudaError_t launch_chain(const Geometry& g, const Group& gr, const Scratch& sc, int l0, int ncall, cudaStream_t st,
                         int priority, bool programmatic) {
    ChainArgs a{};
    a.G = g;
    a.cu = gr.io[0].cu;
    a.state = gr.io[0].state;
    a.refused = sc.refused;
    a.err = sc.err;
    a.l0 = l0;
    a.nl = gr.nl;
    a.ncall = ncall;
    for (int l = 0; l < gr.nl; ++l) a.sl[l] = gr.sl[l];
    programmatic = programmatic && l0 == 0;   // else the launch before writes the state that this one reads early
    return g.ada ? launch_for<true>(g, a, st, priority, programmatic) : launch_for<false>(g, a, st, priority, programmatic);
}

}  // namespace kvec
